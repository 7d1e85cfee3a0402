// FP32 coarse stencil with N = 8 dofs per site, a warp per site: the loads and the reduction that
// the coarse apply and the fused MR iteration share.
//
// Lane = 4 q + rp: rows 2 rp and 2 rp + 1 of column q of every direction's 8 x 8 block, one 16-byte
// load per direction, so a warp reads each 512-byte block in one instruction (with 8-byte loads of
// one row, 10 per thread, the loads' issue and their index arithmetic bounded the kernel: 690
// instructions per warp and site). At 256 x 192 sites (126 MB of blocks) the apply takes 23 us (39
// before), an MR iteration 34 us (121 before, 92 with the capped grid of mr.cuh). The q sum is a
// reduce-scatter: 4 shuffles, after which a lane holds one real number of the result.
#pragma once

#include "common.cuh"

namespace mg {

struct Site8 {
  int nb[5];  // self, +0, -0, +1, -1
  __device__ __forceinline__ Site8(int j, int L0, int L1) {
    const int x1 = j / L0, x0 = j - x1 * L0, row = x1 * L0;
    nb[0] = j;
    nb[1] = row + (x0 + 1 == L0 ? 0 : x0 + 1);
    nb[2] = row + (x0 == 0 ? L0 - 1 : x0 - 1);
    nb[3] = (x1 + 1 == L1 ? 0 : row + L0) + x0;
    nb[4] = (x1 == 0 ? (L1 - 1) * L0 : row - L0) + x0;
  }
};

struct Lane8 {
  int rp, q, row, im;  // rows of the products; row and component (0 re, 1 im) of the lane's result
  bool writes;         // two lanes hold each number: the one that writes it
  __device__ __forceinline__ Lane8() {
    const int lane = threadIdx.x & 31;
    rp = lane & 3;
    q = lane >> 2;
    row = 2 * rp + (lane >> 4);
    im = (lane >> 3) & 1;
    writes = (lane & 4) == 0;
  }
};

__device__ __forceinline__ void load_blocks8(const Cx<float> *__restrict__ Y, int j, const Lane8 &l, float4 (&y)[5]) {
  const float4 *p = reinterpret_cast<const float4 *>(Y + (long long)j * 320) + l.q * 4 + l.rp;
#pragma unroll
  for (int d = 0; d < 5; ++d) y[d] = __ldg(p + d * 32);
}

__device__ __forceinline__ float2 load_col8(const Cx<float> *v, int site, int k) {
  return *reinterpret_cast<const float2 *>(v + (long long)site * 8 + k);
}

// component l.im of row l.row of sum_d Y_d w_d (whole warp)
__device__ __forceinline__ float stencil8(const float4 (&y)[5], const float2 (&w)[5], const Lane8 &l) {
  float a0 = 0.f, a1 = 0.f, b0 = 0.f, b1 = 0.f;
#pragma unroll
  for (int d = 0; d < 5; ++d) {
    a0 = fmaf(y[d].x, w[d].x, a0);
    a1 = fmaf(y[d].x, w[d].y, a1);
    b0 = fmaf(y[d].z, w[d].x, b0);
    b1 = fmaf(y[d].z, w[d].y, b1);
    a0 = fmaf(-y[d].y, w[d].y, a0);
    a1 = fmaf(y[d].y, w[d].x, a1);
    b0 = fmaf(-y[d].w, w[d].y, b0);
    b1 = fmaf(y[d].w, w[d].x, b1);
  }
  const bool up = (l.row & 1) != 0;
  float k0 = up ? b0 : a0, k1 = up ? b1 : a1;
  k0 += __shfl_xor_sync(0xffffffffu, up ? a0 : b0, 16);
  k1 += __shfl_xor_sync(0xffffffffu, up ? a1 : b1, 16);
  float k = l.im ? k1 : k0;
  k += __shfl_xor_sync(0xffffffffu, l.im ? k0 : k1, 8);
  k += __shfl_xor_sync(0xffffffffu, k, 4);
  return k;
}

}  // namespace mg
