// Kernels of the learned near-null setup: a gauge-covariant parallel-transport network
// that maps random spinor fields to Nv near-null vector candidates (replacing most of the
// null-space relaxation of Eq. relax and the adaptive passes), its training by
// backpropagation of a rotation-invariant block loss, and Adam.
//
// Network (per site x, channel-spin index l = 2 c + s, directions self, +0, -0, +1, -1):
//   a_x = sum_dir W_dir T_dir(h)_x,  T_self h_x = h_x, T_{+mu} h_x = U_x^mu h_{x+mu},
//   T_{-mu} h_x = conj(U_{x-mu}^mu) h_{x-mu};   hidden layers h = a / sqrt(1 + |a_c|^2)
// per channel c (both spin components), last layer linear. The weights act on channel and
// spin only, so every layer commutes with U(1) gauge transformations.
//
// Layouts: activations h[f][x][2 C] as bfloat16 pairs (re, im); pre-activations and
// gradients float2 [f][x][2 C]; links float2 [f][x][2]; weights float2 [5][2 co][2 ci].
#include <cuda_bf16.h>

#include "nullnet.h"

namespace mg {

namespace {

// the roundings are spelled out: a transported input that moves by one bit can move the bfloat16
// activation behind it by 2^-9, so every kernel that transports must round alike
__device__ __forceinline__ float2 cmulf(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -__fmul_rn(a.y, b.y)), fmaf(a.x, b.y, __fmul_rn(a.y, b.x)));
}
__device__ __forceinline__ float norm2f(float2 a) { return fmaf(a.x, a.x, __fmul_rn(a.y, a.y)); }
// acc += a * b
__device__ __forceinline__ void cmacf(float2 &acc, float2 a, float2 b) {
  acc.x = fmaf(a.x, b.x, acc.x);
  acc.x = fmaf(-a.y, b.y, acc.x);
  acc.y = fmaf(a.x, b.y, acc.y);
  acc.y = fmaf(a.y, b.x, acc.y);
}
// acc += conj(a) * b
__device__ __forceinline__ void cmacf_conj(float2 &acc, float2 a, float2 b) {
  acc.x = fmaf(a.x, b.x, acc.x);
  acc.x = fmaf(a.y, b.y, acc.x);
  acc.y = fmaf(a.x, b.y, acc.y);
  acc.y = fmaf(-a.y, b.x, acc.y);
}
__device__ __forceinline__ float2 conjf2(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ float2 bf2f(__nv_bfloat162 v) {
  return make_float2(__bfloat162float(v.x), __bfloat162float(v.y));
}
__device__ __forceinline__ __nv_bfloat162 f2bf(float2 v) {
  __nv_bfloat162 r;
  r.x = __float2bfloat16_rn(v.x);
  r.y = __float2bfloat16_rn(v.y);
  return r;
}

// neighbour site and transport phase of direction dir for the forward operator at x:
// T_dir h_x = phase * h_{nb}
__device__ __forceinline__ void fwd_hop(int dir, int x0, int x1, int L0, int L1, const float2 *Uf, long long &nb,
                                        float2 &ph) {
  const long long x = x0 + (long long)L0 * x1;
  switch (dir) {
    case 0: nb = x; ph = make_float2(1.f, 0.f); break;
    case 1: nb = (x0 + 1 == L0 ? 0 : x0 + 1) + (long long)L0 * x1; ph = Uf[2 * x]; break;
    case 2: {
      nb = (x0 == 0 ? L0 - 1 : x0 - 1) + (long long)L0 * x1;
      ph = conjf2(Uf[2 * nb]);
      break;
    }
    case 3: nb = x0 + (long long)L0 * (x1 + 1 == L1 ? 0 : x1 + 1); ph = Uf[2 * x + 1]; break;
    default: {
      nb = x0 + (long long)L0 * (x1 == 0 ? L1 - 1 : x1 - 1);
      ph = conjf2(Uf[2 * nb + 1]);
      break;
    }
  }
}

// adjoint: the contribution of direction dir to dL/dh^*_z comes from site src with phase
// (T_{+mu}: src = z - mu, conj(U_{z-mu}^mu); T_{-mu}: src = z + mu, U_z^mu)
__device__ __forceinline__ void adj_hop(int dir, int z0, int z1, int L0, int L1, const float2 *Uf, long long &src,
                                        float2 &ph) {
  const long long z = z0 + (long long)L0 * z1;
  switch (dir) {
    case 0: src = z; ph = make_float2(1.f, 0.f); break;
    case 1: {
      src = (z0 == 0 ? L0 - 1 : z0 - 1) + (long long)L0 * z1;
      ph = conjf2(Uf[2 * src]);
      break;
    }
    case 2: src = (z0 + 1 == L0 ? 0 : z0 + 1) + (long long)L0 * z1; ph = Uf[2 * z]; break;
    case 3: {
      src = z0 + (long long)L0 * (z1 == 0 ? L1 - 1 : z1 - 1);
      ph = conjf2(Uf[2 * src + 1]);
      break;
    }
    default: src = z0 + (long long)L0 * (z1 + 1 == L1 ? 0 : z1 + 1); ph = Uf[2 * z + 1]; break;
  }
}

// ---------------------------------------------------------------------------
// The transported convolution as a tiled product: for a tile of S sites and one direction the
// transported inputs v_x[k] = phase_x in_{nb(x)}[k] are staged in shared memory (site fastest), the
// weights of all directions once per CTA, and a thread accumulates the spin rows of two channels at SP sites: with
// SP = 4 two 16-byte loads of weights and two of inputs for 16 complex multiply-adds, whose 64 instructions take
// as long as the loads' 16 cycles of shared memory (with one channel 12 cycles of loads met 8 of arithmetic). A thread
// stages one site: its neighbour and phase are worked out once per direction, for all of its channels, and the
// entries are requested while the direction before is multiplied.
// FP32 issue bounds it (150 us of multiply-adds per layer at 16 fields of 128^2, 32 entries): 271 us forward, 264 us
// for the adjoint; with one channel to a thread and a neighbour per entry 328 and 312, with a warp per site, a lane
// per output row and two shuffles per input 2.1 and 2.5 ms. A whole gradient with the loss and weight kernels below:
// 22.1 ms then, 3.8 now. Every output sums its terms in the order direction, input, as fused multiply-adds, so the
// values that are rounded to bfloat16 do not depend on the tiling.
// ---------------------------------------------------------------------------
enum class Conv {
  kHidden,  // bf16 in; gated bf16 out, pre-activation out if asked for
  kLast,    // bf16 in; float2 out
  kAdjoint  // float2 in (dL/da^* of the layer), conj(W)^T, adjoint hops; dL/da^* of the layer before (through its gate)
};

constexpr int kConvThreads = 256;
constexpr int kAhead = 8;  // channels of a thread's site: 32 / 2 entries over at least two rows of threads, or 16 / 2

// sites of a tile for c2 pairs of output channels, SP sites to a thread and kin inputs; a thread stages one site, so
// a tile has at most kConvThreads, and half of them where a thread would stage more than kAhead channels
__host__ __device__ inline int conv_tile(int c2, int sp, int kin) {
  const int s = kConvThreads / c2 * sp, most = kin <= 2 * kAhead ? kConvThreads : kConvThreads / 2;
  return s < most ? s : most;
}

// the two spin entries of a channel as they are stored
template <typename TI>
struct RawPair {
  using T = uint2;
};
template <>
struct RawPair<float2> {
  using T = float4;
};
__device__ __forceinline__ void unpack(uint2 w, float2 &a, float2 &b) {
  a = bf2f(*reinterpret_cast<const __nv_bfloat162 *>(&w.x));
  b = bf2f(*reinterpret_cast<const __nv_bfloat162 *>(&w.y));
}
__device__ __forceinline__ void unpack(float4 w, float2 &a, float2 &b) {
  a = make_float2(w.x, w.y);
  b = make_float2(w.z, w.w);
}

// kin / kout: channel-spin entries (even, at most 32) of the input and output of this product
template <Conv M, typename TI, int SP>
__global__ void __launch_bounds__(kConvThreads, 2) ptconv_kernel(const TI *__restrict__ in, const float2 *__restrict__ U,
                                                              const int *__restrict__ fmap,
                                                              const float2 *__restrict__ W, int kin, int kout, int L0,
                                                              int L1, const float2 *__restrict__ a_prev,
                                                              float2 *__restrict__ a_out,
                                                              __nv_bfloat162 *__restrict__ h_out) {
  using Raw = typename RawPair<TI>::T;
  extern __shared__ float4 conv_smem[];
  const int C = kout / 2, C2 = (C + 1) / 2, S = conv_tile(C2, SP, kin), V = L0 * L1, f = blockIdx.y;
  // [dir][k][channel parity][pair][spin]: a quarter warp's 16-byte loads are consecutive; zero past the last channel
  float2 *Ws = reinterpret_cast<float2 *>(conv_smem);
  float2 *Vs = Ws + 5 * kin * 4 * C2;  // [k][S]
  for (int q = threadIdx.x; q < 5 * kin * 4 * C2; q += kConvThreads) {
    const int dk = q / (4 * C2), r = q - dk * 4 * C2, half = r / (2 * C2);
    const int o = 4 * ((r - half * 2 * C2) >> 1) + 2 * half + (r & 1);
    float2 w = make_float2(0.f, 0.f);
    if (o < kout) {
      if (M == Conv::kAdjoint) {  // W[dir][k][out]: rows of the layer's weights are this product's inputs
        w = conjf2(W[dk * kout + o]);
      } else {  // W[dir][out][k]
        const int dir = dk / kin, k = dk - dir * kin;
        w = W[(dir * kout + o) * kin + k];
      }
    }
    Ws[q] = w;
  }
  const float2 *Uf = U + (size_t)(fmap ? fmap[f] : f) * 2 * V;
  in += (size_t)f * V * kin;
  const int c2 = threadIdx.x % C2, grp = threadIdx.x / C2;
  const bool works = grp * SP < S;
  // staging: this thread's site of the tile and its channels row, row + rows, ...
  const int rows = kConvThreads / S, ss = threadIdx.x % S, row = threadIdx.x / S;
  Raw raw[kAhead];
  float2 ph;
  int y0 = 0, y1 = 0;
  bool there = false;
  auto ahead = [&](int x0, int dir) {
    if (dir == 0) {
      const int x = x0 + ss;
      there = row < rows && x < V;
      y1 = x / L0;
      y0 = x - y1 * L0;
    }
    ph = make_float2(0.f, 0.f);
    long long nb = 0;
    if (there) {
      if (M == Conv::kAdjoint)
        adj_hop(dir, y0, y1, L0, L1, Uf, nb, ph);
      else
        fwd_hop(dir, y0, y1, L0, L1, Uf, nb, ph);
    }
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int ch = row + u * rows;
      raw[u] = Raw{};
      if (there && ch < kin / 2) raw[u] = *reinterpret_cast<const Raw *>(in + nb * kin + 2 * ch);
    }
  };
  ahead(blockIdx.x * S, 0);
  for (int x0 = blockIdx.x * S; x0 < V; x0 += gridDim.x * S) {
    float2 acc[SP][4];
#pragma unroll
    for (int s = 0; s < SP; ++s)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[s][e] = make_float2(0.f, 0.f);
    for (int dir = 0; dir < 5; ++dir) {
      __syncthreads();
#pragma unroll
      for (int u = 0; u < kAhead; ++u) {
        const int ch = row + u * rows;
        if (row < rows && ch < kin / 2) {
          float2 a, b;
          unpack(raw[u], a, b);
          Vs[2 * ch * S + ss] = cmulf(ph, a);
          Vs[(2 * ch + 1) * S + ss] = cmulf(ph, b);
        }
      }
      __syncthreads();
      if (dir < 4)
        ahead(x0, dir + 1);
      else
        ahead(x0 + gridDim.x * S, 0);
      if (works) {
        const float4 *wp = reinterpret_cast<const float4 *>(Ws + dir * kin * 4 * C2) + c2;
        const float4 *vp = reinterpret_cast<const float4 *>(Vs) + grp * (SP / 2);
#pragma unroll 4
        for (int k = 0; k < kin; ++k) {
          const float4 w0 = wp[k * 2 * C2], w1 = wp[k * 2 * C2 + C2];
          const float2 w[4] = {make_float2(w0.x, w0.y), make_float2(w0.z, w0.w), make_float2(w1.x, w1.y),
                               make_float2(w1.z, w1.w)};
          float2 v[SP];
#pragma unroll
          for (int s = 0; s < SP; s += 2) {
            const float4 t = vp[k * (S / 2) + s / 2];
            v[s] = make_float2(t.x, t.y);
            v[s + 1] = make_float2(t.z, t.w);
          }
#pragma unroll
          for (int s = 0; s < SP; ++s)
#pragma unroll
            for (int e = 0; e < 4; ++e) cmacf(acc[s][e], w[e], v[s]);
        }
      }
    }
    if (!works) continue;
#pragma unroll
    for (int s = 0; s < SP; ++s) {
      const int x = x0 + grp * SP + s;
      if (x >= V) break;
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        if (2 * c2 + half >= C) break;
        const float2 p = acc[s][2 * half], q = acc[s][2 * half + 1];
        const size_t o = ((size_t)f * V + x) * kout + 4 * c2 + 2 * half;
        if (M == Conv::kAdjoint) {
          const float4 a = *reinterpret_cast<const float4 *>(a_prev + o);
          const float sq = (a.x * a.x + a.y * a.y) + (a.z * a.z + a.w * a.w);
          const float re = (a.x * p.x + a.y * p.y) + (a.z * q.x + a.w * q.y);
          const float g = rsqrtf(1.f + sq);
          const float dg2 = -g * g * g * re;  // 2 g'(s) Re(a^dagger gh), g' = -g^3 / 2
          *reinterpret_cast<float4 *>(a_out + o) =
              make_float4(g * p.x + dg2 * a.x, g * p.y + dg2 * a.y, g * q.x + dg2 * a.z, g * q.y + dg2 * a.w);
        } else {
          if (M == Conv::kLast || a_out != nullptr)
            *reinterpret_cast<float4 *>(a_out + o) = make_float4(p.x, p.y, q.x, q.y);
          if (M == Conv::kHidden) {
            const float s0 = norm2f(p), s1 = norm2f(q);
            const float g = rsqrtf(1.f + (s0 + s1));
            __nv_bfloat162 h[2] = {f2bf(make_float2(p.x * g, p.y * g)), f2bf(make_float2(q.x * g, q.y * g))};
            *reinterpret_cast<uint2 *>(h_out + o) = *reinterpret_cast<const uint2 *>(h);
          }
        }
      }
    }
  }
}

// Per-CTA partial sums of dL/dW^*[dir][lo][li] = sum_x ga_x[lo] conj(T_dir h_x[li]) over a
// contiguous range of (field, site) pairs; partials[cta][entry] (entry = (dir co2 + lo) ci2 + li)
// A thread owns input entry li (its lane) and output rows lo0 .. lo0 + 3 of every direction: per staged
// site two 16-byte broadcast loads of g and five loads of T h for 20 complex multiply-adds. The next group's
// rows are requested while this one's are multiplied (16 fields of 128^2, 32 entries: 361 -> 261 us; eight rows to a
// thread with 4 warps to a CTA took 300 us).
constexpr int kWG = 16;  // sites staged per group
__global__ void __launch_bounds__(256, 2) ptconv_bwd_weight_kernel(const float2 *__restrict__ ga,
                                                                   const __nv_bfloat162 *__restrict__ h_in,
                                                                   const float2 *__restrict__ U,
                                                                   const int *__restrict__ fmap, int nf, int ci2,
                                                                   int co2, int L0, int L1,
                                                                   float2 *__restrict__ partials) {
  __shared__ float2 gs[kWG][32];
  __shared__ float2 Ts[kWG][5][32];
  const long long V = (long long)L0 * L1, total = V * nf;
  const long long per = (total + gridDim.x - 1) / gridDim.x;
  const long long p0 = (long long)blockIdx.x * per, p1 = p0 + per < total ? p0 + per : total;
  const int ne = 5 * co2 * ci2;
  float2 acc[5][4];
#pragma unroll
  for (int d = 0; d < 5; ++d)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[d][e] = make_float2(0.f, 0.f);
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // warp w stages sites g0 + w, g0 + w + 8: the gradient row and the five transported inputs, requested a group
  // ahead
  float2 gv[2], ph[2][5];
  __nv_bfloat162 hv[2][5];
  auto request = [&](long long g0) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const long long p = g0 + wid + 8 * u;
      gv[u] = make_float2(0.f, 0.f);
#pragma unroll
      for (int d = 0; d < 5; ++d) {
        ph[u][d] = make_float2(0.f, 0.f);
        hv[u][d] = f2bf(ph[u][d]);
      }
      if (p < p1) {
        const int f = (int)(p / V);
        const int x = (int)(p - (long long)f * V);
        const int x1 = x / L0, x0 = x - x1 * L0;
        const float2 *Uf = U + (size_t)(fmap ? fmap[f] : f) * 2 * V;
        if (lane < co2) gv[u] = ga[(size_t)p * co2 + lane];
#pragma unroll
        for (int d = 0; d < 5; ++d) {
          long long nb;
          fwd_hop(d, x0, x1, L0, L1, Uf, nb, ph[u][d]);
          if (lane < ci2) hv[u][d] = h_in[((size_t)f * V + nb) * ci2 + lane];
        }
      }
    }
  };
  request(p0);
  for (long long g0 = p0; g0 < p1; g0 += kWG) {
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int s = wid + 8 * u;
      gs[s][lane] = gv[u];
#pragma unroll
      for (int d = 0; d < 5; ++d) Ts[s][d][lane] = cmulf(ph[u][d], bf2f(hv[u][d]));
    }
    __syncthreads();
    request(g0 + kWG);
    if (4 * wid < co2) {
#pragma unroll 4
      for (int s = 0; s < kWG; ++s) {
        const float4 g01 = *reinterpret_cast<const float4 *>(&gs[s][4 * wid]);
        const float4 g23 = *reinterpret_cast<const float4 *>(&gs[s][4 * wid + 2]);
        const float2 g[4] = {make_float2(g01.x, g01.y), make_float2(g01.z, g01.w), make_float2(g23.x, g23.y),
                             make_float2(g23.z, g23.w)};
#pragma unroll
        for (int d = 0; d < 5; ++d) {
          const float2 t = Ts[s][d][lane];
#pragma unroll
          for (int e = 0; e < 4; ++e) cmacf_conj(acc[d][e], t, g[e]);
        }
      }
    }
  }
  if (lane < ci2) {
#pragma unroll
    for (int d = 0; d < 5; ++d)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int lo = 4 * wid + e;
        if (lo < co2) partials[(size_t)blockIdx.x * ne + (d * co2 + lo) * ci2 + lane] = acc[d][e];
      }
  }
}

// gW[q] = sum over CTAs of partials[cta][q] (fixed order, FP64 sums): a block takes 32 entries, warp w the
// CTAs w, w + 8, ... (a thread per entry walked all of them alone, 95 us of latency per layer)
__global__ void __launch_bounds__(256) sum_partials_kernel(const float2 *__restrict__ partials, int nparts, int ne,
                                                           float2 *__restrict__ gW) {
  __shared__ double2 sh[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, q = blockIdx.x * 32 + lane;
  double re = 0.0, im = 0.0;
  if (q < ne) {
#pragma unroll 4
    for (int c = w; c < nparts; c += 8) {
      const float2 v = partials[(size_t)c * ne + q];
      re += v.x;
      im += v.y;
    }
  }
  sh[w][lane] = make_double2(re, im);
  __syncthreads();
  if (w != 0 || q >= ne) return;
#pragma unroll
  for (int k = 1; k < 8; ++k) {
    re += sh[k][lane].x;
    im += sh[k][lane].y;
  }
  gW[q] = make_float2((float)re, (float)im);
}

// Rotation-invariant block loss and dL/dy^*, four blocks per warp. G = W^dagger W and C = W^dagger V in
// FP32 (a lane forms two entries of each over the block's rows, staged in shared memory), then the small
// dense algebra in FP64: G = L L^dagger (a relative ridge of 1e-7 tr G / nv keeps FP32 round-off from
// breaking it), A = G^{-1} C, L_b = nv - Re tr(C^dagger A); grad = -(V - W A) A^dagger. Eight lanes share
// a block's FP64 work (row i of L, then column i of A), so a warp's FP64 instructions, which bound the
// kernel, serve four blocks: 232 us for 16 fields of 128^2 (216 with the FP32 sums in a chain); a serial factorisation
// by one lane per warp and block took 2.2 ms.
constexpr int kMaxNv = 8;
constexpr int kLossWarps = 4, kLossBlocks = 4;
struct LossSmem {
  float2 w[32][kMaxNv + 1], v[32][kMaxNv + 1];  // rows of the block in work
  double2 G[kLossBlocks][kMaxNv * kMaxNv];      // G, then L below the diagonal
  double2 C[kLossBlocks][kMaxNv * kMaxNv];
  float2 A[kLossBlocks][kMaxNv * kMaxNv];
};

// A lane's four sums over 2^LEVEL rows, from `first` on and 32 / 2^LEVEL apart (LEVEL 5: all rows), as a tree of
// additions: five roundings on the way of a product, where a chain over the rows has up to 32.
template <int LEVEL>
__device__ __forceinline__ void loss_sums(const LossSmem &sm, int first, int rows, int k, int j, float2 &g0, float2 &g1,
                                          float2 &c0, float2 &c1) {
  if constexpr (LEVEL == 0) {
    g0 = g1 = c0 = c1 = make_float2(0.f, 0.f);
    if (first < rows) {
      const float2 a = sm.w[first][k], e = sm.w[first][k + 4], wj = sm.w[first][j], vj = sm.v[first][j];
      cmacf_conj(g0, a, wj);
      cmacf_conj(g1, e, wj);
      cmacf_conj(c0, a, vj);
      cmacf_conj(c1, e, vj);
    }
  } else {
    float2 h0, h1, d0, d1;
    loss_sums<LEVEL - 1>(sm, first, rows, k, j, g0, g1, c0, c1);
    loss_sums<LEVEL - 1>(sm, first + (32 >> LEVEL), rows, k, j, h0, h1, d0, d1);
    g0 = make_float2(g0.x + h0.x, g0.y + h0.y);
    g1 = make_float2(g1.x + h1.x, g1.y + h1.y);
    c0 = make_float2(c0.x + d0.x, c0.y + d0.y);
    c1 = make_float2(c1.x + d1.x, c1.y + d1.y);
  }
}

__global__ void __launch_bounds__(32 * kLossWarps) nullnet_loss_kernel(const float2 *__restrict__ y,
                                                                       const float2 *__restrict__ target,
                                                                       const int *__restrict__ fmap, int nv,
                                                                       BlockGeo bg, float scale,
                                                                       float2 *__restrict__ gy,
                                                                       double *__restrict__ lossb) {
  extern __shared__ float4 loss_smem[];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  LossSmem &sm = reinterpret_cast<LossSmem *>(loss_smem)[wid];
  const int f = blockIdx.y;
  const long long V = (long long)bg.L0 * bg.L1;
  const long long first = ((long long)blockIdx.x * kLossWarps + wid) * kLossBlocks;
  const int count = bg.nblocks - first < kLossBlocks ? (int)(bg.nblocks - first) : kLossBlocks;
  if (count <= 0) return;  // whole warps leave together
  const int rows = bg.bvol * 2, sp = lane & 1;
  const bool act = lane < rows;
  const float2 *yf = y + (size_t)f * V * 2 * nv;
  const float2 *tf = target + (size_t)(fmap ? fmap[f] : f) * nv * V * 2;
  const float2 zero = make_float2(0.f, 0.f);
  // entries [lane] and [lane + 32] of each block's G and C
  for (int b = 0; b < count; ++b) {
    const long long site = act ? fine_site_of(bg, first + b, lane >> 1) : 0;
    __syncwarp();
#pragma unroll
    for (int k = 0; k < kMaxNv; ++k) {
      sm.w[lane][k] = (act && k < nv) ? yf[(size_t)site * 2 * nv + 2 * k + sp] : zero;
      sm.v[lane][k] = (act && k < nv) ? tf[((size_t)k * V + site) * 2 + sp] : zero;
    }
    __syncwarp();
    const int k0 = lane >> 3, j = lane & 7;
    float2 g0, g1, c0, c1;
    loss_sums<5>(sm, 0, rows, k0, j, g0, g1, c0, c1);
    // unused vectors: an identity block, so that the factorisation runs over all eight rows
    const bool in0 = k0 < nv && j < nv, in1 = k0 + 4 < nv && j < nv;
    sm.G[b][lane] = in0 ? make_double2(g0.x, g0.y) : make_double2(k0 == j ? 1.0 : 0.0, 0.0);
    sm.G[b][lane + 32] = in1 ? make_double2(g1.x, g1.y) : make_double2(k0 + 4 == j ? 1.0 : 0.0, 0.0);
    sm.C[b][lane] = make_double2(c0.x, c0.y);
    sm.C[b][lane + 32] = make_double2(c1.x, c1.y);
  }
  __syncwarp();
  {
    const int q = lane >> 3, i = lane & 7;  // block of the warp; row of L and column of A
    const bool mine = q < count;
    const int b = mine ? q : 0;  // idle lanes shadow block 0 and write nothing
    double2 *G = sm.G[b], *C = sm.C[b];
    double tr = 0.0;
    for (int k = 0; k < nv; ++k) tr += G[k * kMaxNv + k].x;
    const double ridge = 1e-7 * tr / nv + 1e-30;
    double rinv[kMaxNv];
    double2 L[kMaxNv];  // row i of L
#pragma unroll
    for (int j = 0; j < kMaxNv; ++j) {
      // L_ij = (G_ij - sum_k L_ik conj(L_jk)) / L_jj, G_ij = conj(G_ji) read from the upper part
      double re = G[j * kMaxNv + i].x, im = -G[j * kMaxNv + i].y;
      if (i == j) re += ridge;
#pragma unroll
      for (int k = 0; k < j; ++k) {
        const double2 ljk = G[j * kMaxNv + k];
        re = fma(-L[k].x, ljk.x, fma(-L[k].y, ljk.y, re));
        im = fma(-L[k].y, ljk.x, fma(L[k].x, ljk.y, im));
      }
      const double d = sqrt(fmax(__shfl_sync(0xffffffffu, re, 8 * q + j), 1e-300));
      rinv[j] = 1.0 / d;
      L[j] = make_double2(re * rinv[j], im * rinv[j]);
      __syncwarp();
      if (mine && i > j) G[i * kMaxNv + j] = L[j];
      __syncwarp();
    }
    // column i of A = G^{-1} C: L u = c, then L^dagger a = u
    double2 u[kMaxNv];
#pragma unroll
    for (int r = 0; r < kMaxNv; ++r) {
      double re = C[r * kMaxNv + i].x, im = C[r * kMaxNv + i].y;
#pragma unroll
      for (int k = 0; k < r; ++k) {
        const double2 l = G[r * kMaxNv + k];
        re = fma(-l.x, u[k].x, fma(l.y, u[k].y, re));
        im = fma(-l.x, u[k].y, fma(-l.y, u[k].x, im));
      }
      u[r] = make_double2(re * rinv[r], im * rinv[r]);
    }
    double t = 0.0;  // Re tr(C^dagger A) = sum_ij Re(conj(C_ij) A_ij)
#pragma unroll
    for (int r = kMaxNv - 1; r >= 0; --r) {
      double re = u[r].x, im = u[r].y;
#pragma unroll
      for (int k = r + 1; k < kMaxNv; ++k) {
        const double2 l = G[k * kMaxNv + r];  // (L^dagger)_rk = conj(L_kr)
        re = fma(-l.x, u[k].x, fma(-l.y, u[k].y, re));
        im = fma(-l.x, u[k].y, fma(l.y, u[k].x, im));
      }
      u[r] = make_double2(re * rinv[r], im * rinv[r]);
      t = fma(C[r * kMaxNv + i].x, u[r].x, fma(C[r * kMaxNv + i].y, u[r].y, t));
      if (mine) sm.A[b][r * kMaxNv + i] = make_float2((float)u[r].x, (float)u[r].y);
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (mine && i == 0) lossb[(size_t)f * bg.nblocks + first + b] = (double)nv - t;
  }
  __syncwarp();
  if (!act) return;
  float2 *gf = gy + (size_t)f * V * 2 * nv;
  for (int b = 0; b < count; ++b) {
    const long long site = fine_site_of(bg, first + b, lane >> 1);
    const float2 *A = sm.A[b];
    float2 w[kMaxNv], r[kMaxNv];
#pragma unroll
    for (int k = 0; k < kMaxNv; ++k) {
      w[k] = k < nv ? yf[(size_t)site * 2 * nv + 2 * k + sp] : zero;
      r[k] = k < nv ? tf[((size_t)k * V + site) * 2 + sp] : zero;
    }
    // R = V - W A, grad_k' = -sum_k R_k conj(A_k'k)
#pragma unroll
    for (int k = 0; k < kMaxNv; ++k)
#pragma unroll
      for (int q = 0; q < kMaxNv; ++q) cmacf(r[k], make_float2(-w[q].x, -w[q].y), A[q * kMaxNv + k]);
#pragma unroll
    for (int kp = 0; kp < kMaxNv; ++kp) {
      if (kp >= nv) break;
      float2 t = zero;
#pragma unroll
      for (int k = 0; k < kMaxNv; ++k) cmacf(t, r[k], conjf2(A[kp * kMaxNv + k]));
      gf[(size_t)site * 2 * nv + 2 * kp + sp] = make_float2(-scale * t.x, -scale * t.y);
    }
  }
}

// Adam on the real and imaginary parts (the real-parameter gradient is 2 (Re, Im) of dL/dW^*)
__global__ void adam_kernel(float *__restrict__ w, const float *__restrict__ g, float *__restrict__ m1,
                            float *__restrict__ m2, long long n, float lr, float b1, float b2, float c1, float c2,
                            float eps) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = 2.f * g[i];
  const float a = b1 * m1[i] + (1.f - b1) * gi;
  const float b = b2 * m2[i] + (1.f - b2) * gi * gi;
  m1[i] = a;
  m2[i] = b;
  w[i] -= lr * (a / c1) / (sqrtf(b / c2) + eps);
}

// noise [c][f][x][2] complex128 (Philox Gaussians) -> bf16 [f][x][2 c + s]
__global__ void pack_noise_kernel(const Cx<double> *__restrict__ z, int cin, long long V, int nf,
                                  __nv_bfloat162 *__restrict__ h) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long n = (long long)nf * V * 2 * cin;
  if (i >= n) return;
  const int l = (int)(i % (2 * cin));
  const long long fx = i / (2 * cin);
  const int c = l >> 1, s = l & 1;
  const Cx<double> v = z[((size_t)c * nf * V + fx) * 2 + s];
  h[i] = f2bf(make_float2((float)v.re, (float)v.im));
}

// predicted vectors y[x][2 nv] (float2) -> v[k][x][2] complex128 (the layout of the setup's vectors)
__global__ void unpack_vectors_kernel(const float2 *__restrict__ y, int nv, long long V,
                                      Cx<double> *__restrict__ out) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)nv * V * 2) return;
  const int s = (int)(i & 1);
  const long long kx = i >> 1;
  const int k = (int)(kx / V);
  const long long x = kx - (long long)k * V;
  const float2 v = y[(size_t)x * 2 * nv + 2 * k + s];
  out[i] = mk((double)v.x, (double)v.y);
}

// complex128 -> float2 (links, targets)
__global__ void to_float2_kernel(const Cx<double> *__restrict__ a, long long n, float2 *__restrict__ b) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) b[i] = make_float2((float)a[i].re, (float)a[i].im);
}

int blocks_for(long long n, int t) { return (int)((n + t - 1) / t); }

template <Conv M, typename TI, int SP>
void conv_launch_tile(const TI *in, const float2 *U, const int *fmap, const float2 *W, int kin, int kout, int L0,
                      int L1, int nf, const float2 *a_prev, float2 *a_out, __nv_bfloat162 *h_out, cudaStream_t s) {
  const int c2 = (kout / 2 + 1) / 2, S = conv_tile(c2, SP, kin);
  const auto fn = ptconv_kernel<M, TI, SP>;
  const size_t smem = ((size_t)5 * kin * 4 * c2 + (size_t)kin * S) * sizeof(float2);
  MG_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  // CTAs per field: at most the two resident on each of 152 SMs over all fields (each stages the weights once; a
  // few CTAs more would run a second wave of their own)
  const long long tiles = ((long long)L0 * L1 + S - 1) / S;
  long long gx = 152 * 2 / nf;
  if (gx < 1) gx = 1;
  if (gx > tiles) gx = tiles;
  fn<<<dim3((unsigned int)gx, nf), kConvThreads, smem, s>>>(in, U, fmap, W, kin, kout, L0, L1, a_prev, a_out, h_out);
  MG_LAUNCHED();
}

// four sites to a thread, or two where tiles of the wider form would not give every SM one (a gradient with 32
// entries: one field of 64^2, 32 tiles: 436 us wide, 390 narrow; 128^2, 128 tiles: 524 both; eight fields of 64^2,
// 256 tiles: 734 and 765)
template <Conv M, typename TI>
void conv_launch(const TI *in, const float2 *U, const int *fmap, const float2 *W, int kin, int kout, int L0, int L1,
                 int nf, const float2 *a_prev, float2 *a_out, __nv_bfloat162 *h_out, cudaStream_t s) {
  const int S = conv_tile((kout / 2 + 1) / 2, 4, kin);
  if (((long long)L0 * L1 + S - 1) / S * nf >= 152)
    conv_launch_tile<M, TI, 4>(in, U, fmap, W, kin, kout, L0, L1, nf, a_prev, a_out, h_out, s);
  else
    conv_launch_tile<M, TI, 2>(in, U, fmap, W, kin, kout, L0, L1, nf, a_prev, a_out, h_out, s);
}

}  // namespace

void launch_ptconv_fwd(const void *h_in, const float2 *U, const int *fmap, const float2 *W, int ci2, int co2,
                       int L0, int L1, int nf, bool last, float2 *a_out, void *h_out, cudaStream_t s) {
  const auto *hi = static_cast<const __nv_bfloat162 *>(h_in);
  if (last)
    conv_launch<Conv::kLast>(hi, U, fmap, W, ci2, co2, L0, L1, nf, nullptr, a_out, nullptr, s);
  else
    conv_launch<Conv::kHidden>(hi, U, fmap, W, ci2, co2, L0, L1, nf, nullptr, a_out,
                               static_cast<__nv_bfloat162 *>(h_out), s);
}

void launch_ptconv_bwd_data(const float2 *ga, const float2 *U, const int *fmap, const float2 *W, int ci2, int co2,
                            int L0, int L1, int nf, const float2 *a_prev, float2 *ga_prev, cudaStream_t s) {
  conv_launch<Conv::kAdjoint>(ga, U, fmap, W, co2, ci2, L0, L1, nf, a_prev, ga_prev, nullptr, s);
}

void launch_ptconv_bwd_weight(const float2 *ga, const void *h_in, const float2 *U, const int *fmap, int nf, int ci2,
                              int co2, int L0, int L1, float2 *partials, int nparts, float2 *gW, cudaStream_t s) {
  ptconv_bwd_weight_kernel<<<nparts, 256, 0, s>>>(ga, static_cast<const __nv_bfloat162 *>(h_in), U, fmap, nf, ci2,
                                                  co2, L0, L1, partials);
  MG_LAUNCHED();
  const int ne = 5 * co2 * ci2;
  sum_partials_kernel<<<blocks_for(ne, 32), 256, 0, s>>>(partials, nparts, ne, gW);
  MG_LAUNCHED();
}

void launch_nullnet_loss(const float2 *y, const float2 *target, const int *fmap, int nv, const BlockGeo &bg, int nf,
                         float scale, float2 *gy, double *lossb, cudaStream_t s) {
  const dim3 grid(blocks_for(bg.nblocks, kLossWarps * kLossBlocks), nf);
  const int smem = kLossWarps * (int)sizeof(LossSmem);
  MG_CUDA(cudaFuncSetAttribute(nullnet_loss_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  nullnet_loss_kernel<<<grid, 32 * kLossWarps, smem, s>>>(y, target, fmap, nv, bg, scale, gy, lossb);
  MG_LAUNCHED();
}

void launch_adam(float *w, const float *g, float *m1, float *m2, long long n, float lr, long long t,
                 cudaStream_t s) {
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
  adam_kernel<<<blocks_for(n, 256), 256, 0, s>>>(w, g, m1, m2, n, lr, b1, b2, c1, c2, 1e-8f);
  MG_LAUNCHED();
}

void launch_pack_noise(const Cx<double> *z, int cin, long long V, int nf, void *h, cudaStream_t s) {
  const long long n = (long long)nf * V * 2 * cin;
  pack_noise_kernel<<<blocks_for(n, 256), 256, 0, s>>>(z, cin, V, nf, static_cast<__nv_bfloat162 *>(h));
  MG_LAUNCHED();
}

void launch_unpack_vectors(const float2 *y, int nv, long long V, Cx<double> *out, cudaStream_t s) {
  unpack_vectors_kernel<<<blocks_for((long long)nv * V * 2, 256), 256, 0, s>>>(y, nv, V, out);
  MG_LAUNCHED();
}

void launch_to_float2(const Cx<double> *a, long long n, float2 *b, cudaStream_t s) {
  to_float2_kernel<<<blocks_for(n, 256), 256, 0, s>>>(a, n, b);
  MG_LAUNCHED();
}

}  // namespace mg
