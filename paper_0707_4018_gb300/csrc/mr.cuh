// Reduction helpers of the fused MR smoothing kernels (paper: MR with under-relaxation
// omega as the relaxation method): block trees of the partial sums, and the step length
// alpha = omega <A r, r> / |A r|^2 formed by every block of the consuming launch from the
// producing launch's block partials, in one fixed order.
#pragma once

#include "common.cuh"

namespace mg {

// block-wide sum of NOUT values of type T; the result is valid in thread 0 (sh: 32 NOUT)
template <int NOUT, typename T>
__device__ __forceinline__ void block_reduce(T (&v)[NOUT], T *sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int k = 0; k < NOUT; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
  }
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < NOUT; ++k) sh[wid * NOUT + k] = v[k];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < NOUT; ++k) {
      T t = (T)0;
      for (int w = 0; w < nw; ++w) t += sh[w * NOUT + k];
      v[k] = t;
    }
  }
}

// Blocks of one MR launch per vector; a block strides over the rest of a larger lattice. Every block of
// the next launch sums all of a vector's partials, so one block per 256 units would make that sum
// quadratic in the lattice: at 1024 x 768 it was 60 to 75 % of an iteration (level 0: 45 us with it,
// 11 without; level 1: 121 and 47). Up to 1216 partials (5 loads per thread) it is small beside the rest.
// Solves in ms with 304 / 608 / 1216 / 2432 / 4864 blocks: 512 x 512 20.1 / 20.1 / 22.4 / 24.3 / 24.3,
// 1024 x 768 46.7 / 43.0 / 44.0 / 51.4 / 64.3, 2048 x 1024 111 / 99.0 / 97.7 / 107 / 136; four sources at
// 1024 x 768 199 / 202 / 211 / 243 / 276.
constexpr int kMrGrid = 1216;
inline int mr_blocks(long long full) { return (int)(full < kMrGrid ? full : kMrGrid); }

// Threads per block of the fine-level MR and apply kernels: small lattices take smaller blocks, which
// reach more SMs (64^2 in FP64, bound by the FP64 rate: an MR iteration on 16 of 152 SMs took 16 us).
inline int site_threads(long long sites) { return sites <= 64LL * 152 ? 64 : 256; }

// the warp's sums of v[0], v[1] and v[2], in the lanes with lane & 3 = 0, 1 and 2: the values part over the lanes of a
// group of four first, 6 additions (each holds an FP64 pipe for 16 cycles) where three butterflies take 15
template <typename R>
__device__ __forceinline__ R warp_reduce3(const R (&v)[3]) {
  const bool hi = (threadIdx.x & 2) != 0, odd = (threadIdx.x & 1) != 0;
  const R a = (hi ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, hi ? v[0] : v[2], 2);
  const R b = (hi ? (R)0 : v[1]) + __shfl_xor_sync(0xffffffffu, hi ? v[1] : (R)0, 2);
  R k = (odd ? b : a) + __shfl_xor_sync(0xffffffffu, odd ? a : b, 1);
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
  return k;
}

// sum over the block of the values that lanes 0, 1 and 2 of every warp hold, in threads 0, 1 and 2 (sh: 32 x 3)
template <typename R>
__device__ __forceinline__ R block_sum3(R k, R *sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (lane < 3) sh[wid * 3 + lane] = k;
  __syncthreads();
  R t = (R)0;
  if (threadIdx.x < 3)
    for (int w = 0; w < nw; ++w) t += sh[w * 3 + threadIdx.x];
  return t;
}

// this block's (<A r, r> re, im, |A r|^2) into part_out[3 blockIdx.x ..]
template <typename R>
__device__ __forceinline__ void mr_publish_lanes(R k, R *part_out, R *sh) {
  const R t = block_sum3<R>(k, sh);
  if (threadIdx.x < 3) part_out[3 * blockIdx.x + threadIdx.x] = t;
}
template <typename R>
__device__ __forceinline__ void mr_publish(const R (&v)[3], R *part_out, R *sh) {
  mr_publish_lanes<R>(warp_reduce3<R>(v), part_out, sh);
}

// alpha = omega <A r, r> / |A r|^2 from the `nb` block partials of the previous launch:
// thread t adds blocks t, t + blockDim, ..., then the block tree; thread 0 divides and
// broadcasts. Every thread of the block must call it.
template <typename R>
__device__ __forceinline__ Cx<R> mr_alpha(const R *part_in, int nb, double omega, R *sh) {
  R v[3] = {(R)0, (R)0, (R)0};
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
    v[0] += __ldcg(part_in + 3 * b);
    v[1] += __ldcg(part_in + 3 * b + 1);
    v[2] += __ldcg(part_in + 3 * b + 2);
  }
  const R t = block_sum3<R>(warp_reduce3<R>(v), sh);
  __shared__ R s_alpha[2];
  if (threadIdx.x < 32) {
    const R den = __shfl_sync(0xffffffffu, t, 2);
    if (threadIdx.x < 2) s_alpha[threadIdx.x] = den > (R)0 ? (R)omega * t / den : (R)0;
  }
  __syncthreads();
  return mk(s_alpha[0], s_alpha[1]);
}

template <typename R>
__device__ __forceinline__ Cx<R> mr_step(Cx<R> r, Cx<R> Ar, Cx<R> malpha) {
  cmac(r, malpha, Ar);
  return r;
}

}  // namespace mg
