// Fine Wilson operator on a 4d SU(3) lattice (paper, definition of D following
// Eq. 1, with four spins, three colours and the DeGrand-Rossi gamma basis;
// diagonal d + m = 4 + m, periodic boundaries).
//
// DeGrand-Rossi: every gamma_mu = [[0, A_mu], [A_mu^dagger, 0]] in 2 x 2 spin
// blocks with A_mu unitary, so (1 -+ gamma_mu) has rank two and is fixed by its
// upper half:
//   (1 - gamma_mu) psi = (h, -A_mu^dagger h),  h = psi_up - A_mu psi_dn
//   (1 + gamma_mu) psi = (h,  A_mu^dagger h),  h = psi_up + A_mu psi_dn
// with psi_up = (psi_0, psi_1), psi_dn = (psi_2, psi_3). A hop therefore
// projects the neighbour's spinor to the half spinor h (2 spins x 3 colours),
// applies the colour link to it (18 complex multiply-adds instead of 36) and
// rebuilds the lower spins from the upper ones. The A_mu are
//   mu = 0: [[0, i], [i, 0]]    mu = 1: [[0, -1], [1, 0]]
//   mu = 2: [[i, 0], [0, -i]]   mu = 3: [[1, 0], [0, 1]].
//
// Layouts (site-major, the library's boundary layout): psi[x][s][c] (12 complex,
// 96 B in FP32), U[x][mu][a][b] (4 x 9 complex; U_x^mu links x to x + mu-hat).
// A warp computes 32 consecutive sites, one per lane, hop after hop; the
// neighbours' spinors and the hop's links are gathered by the whole warp in
// contiguous pieces through shared memory. The backward links are the
// neighbours' forward links, so an apply streams psi, U and out from HBM about
// once: 60 complex per site = 480 B (FP32) / 960 B (FP64). The neighbour
// spinors (8 per site) and links (2 reads each) come from L2, which makes the
// on-chip traffic about 3x the HBM traffic.
#include <cstdlib>

#include "kernels.h"
#include "wilson4d.cuh"

namespace mg {

namespace {

// ---------------------------------------------------------------------------
// Warp-cooperative staging. A warp owns 32 consecutive sites. The 96-B spinors
// and 72-B links of its 32 neighbours in one direction are gathered by the
// whole warp in 16-B (spinor) and 8-B (link) pieces, consecutive lanes taking
// consecutive pieces, so every load instruction reads contiguous memory
// wherever the 32 neighbours are consecutive sites (everywhere except at the
// periodic wrap of direction mu). Each thread then reads its own record from
// shared memory. Strides: a staged FP32 spinor takes 7 float4 (112 B), a staged
// FP64 spinor 13 double2 (208 B) and a link 9 complex: conflict-free reads.
// ---------------------------------------------------------------------------
template <typename R>
struct Stage;
template <>
struct Stage<float> {
  using V = float4;                 // one gathered spinor piece (2 complex)
  static constexpr int PIECES = 6;  // pieces per spinor
  static constexpr int STRIDE = 7;  // staged spinor stride in pieces
};
template <>
struct Stage<double> {
  using V = double2;  // one complex
  static constexpr int PIECES = 12;
  static constexpr int STRIDE = 13;
};

// sp[lane] <- spinor of site `site` of lane `lane` (all 32 lanes take part)
template <typename R>
__device__ __forceinline__ void gather_spinors(const Cx<R> *__restrict__ f, int site, int lane,
                                               typename Stage<R>::V *sp) {
  using S = Stage<R>;
  const typename S::V *src = reinterpret_cast<const typename S::V *>(f);
#pragma unroll
  for (int k = 0; k < S::PIECES; ++k) {
    const int c = lane + 32 * k, i = c / S::PIECES, j = c - i * S::PIECES;
    const int si = __shfl_sync(0xffffffffu, site, i);
    sp[i * S::STRIDE + j] = __ldg(src + (long long)si * S::PIECES + j);
  }
}

// lk[lane] <- link mu of site `site` of lane `lane`
template <typename R>
__device__ __forceinline__ void gather_links(const Cx<R> *__restrict__ U, int site, int mu, int lane, Cx<R> *lk) {
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const int c = lane + 32 * k, i = c / 9, j = c - i * 9;
    const int si = __shfl_sync(0xffffffffu, site, i);
    lk[i * 9 + j] = U[((long long)si * 4 + mu) * 9 + j];
  }
}

template <typename R>
__device__ __forceinline__ void read_spinor(const typename Stage<R>::V *sp, int lane, Cx<R> (&p)[12]) {
  using S = Stage<R>;
  const typename S::V *q = sp + lane * S::STRIDE;
  if (sizeof(R) == 4) {
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      const float4 w = *reinterpret_cast<const float4 *>(q + i);
      p[2 * i] = mk((R)w.x, (R)w.y);
      p[2 * i + 1] = mk((R)w.z, (R)w.w);
    }
  } else {
#pragma unroll
    for (int i = 0; i < 12; ++i) {
      const double2 w = *reinterpret_cast<const double2 *>(q + i);
      p[i] = mk((R)w.x, (R)w.y);
    }
  }
}

}  // namespace

constexpr int DSLASH4_WARPS = 4;

// out = a (D in) + c b for vector blockIdx.y of a batch (stride ldv complex); with
// SHIFT the diagonal of that vector is diag + shift[blockIdx.y]
template <typename R, bool SHIFT>
__global__ void __launch_bounds__(32 * DSLASH4_WARPS, sizeof(R) == 4 ? 5 : 2) dslash4_kernel(const Cx<R> *__restrict__ U,
                                                                   const Cx<R> *__restrict__ in,
                                                                   Cx<R> *__restrict__ out, Geo4 g, R diag,
                                                                   const Cx<R> *__restrict__ b, R a, R c,
                                                                   long long ldv,
                                                                   const double *__restrict__ shift) {
  using S = Stage<R>;
  __shared__ typename S::V sp_all[DSLASH4_WARPS][32 * S::STRIDE];
  __shared__ Cx<R> lk_all[DSLASH4_WARPS][32 * 9];
  if (SHIFT) diag += (R)shift[blockIdx.y];
  in += blockIdx.y * ldv;
  out += blockIdx.y * ldv;
  if (b != nullptr) b += blockIdx.y * ldv;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int V = (int)g.nsites;
  const int warp_first = (blockIdx.x * DSLASH4_WARPS + w) * 32;
  if (warp_first >= V) return;  // whole warps leave together
  const int xr = warp_first + lane;
  const bool valid = xr < V;
  const int x = valid ? xr : V - 1;  // tail lanes shadow the last site (no store)
  typename S::V *sp = sp_all[w];
  Cx<R> *lk = lk_all[w];
  // coordinates and strides of this lane's site
  int cc[4], st[4];
  {
    int r = x, stride = 1;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      cc[mu] = mu < 3 ? r % g.L[mu] : r;
      r = mu < 3 ? r / g.L[mu] : 0;
      st[mu] = stride;
      stride *= g.L[mu];
    }
  }
  Cx<R> acc[12];
#pragma unroll
  for (int i = 0; i < 12; ++i) acc[i] = mk((R)0, (R)0);
  // the hops one after another (not unrolled: one hop's loads are not hoisted into
  // another's registers): singly in FP32, whose 96 registers hold no second product, a direction's two
  // together in FP64, where they share additions (16^3 x 32: 224 us, singly 241)
  if constexpr (sizeof(R) == 4) {
#pragma unroll 1
    for (int hop = 0; hop < 8; ++hop) {
      const int mu = hop >> 1;
      int cm = cc[0], sm = st[0], Lm = g.L[0];
      if (mu == 1) { cm = cc[1]; sm = st[1]; Lm = g.L[1]; }
      if (mu == 2) { cm = cc[2]; sm = st[2]; Lm = g.L[2]; }
      if (mu == 3) { cm = cc[3]; sm = st[3]; Lm = g.L[3]; }
      const bool fwd = (hop & 1) == 0;
      const int nb = fwd ? (cm + 1 == Lm ? x - cm * sm : x + sm) : (cm == 0 ? x + (Lm - 1) * sm : x - sm);
      __syncwarp();
      gather_spinors<R>(in, nb, lane, sp);
      gather_links<R>(U, fwd ? x : nb, mu, lane, lk);
      __syncwarp();
      Cx<R> p[12];
      read_spinor<R>(sp, lane, p);
      hop_dispatch<R>(hop, p, lk + lane * 9, acc);
    }
  } else {
#pragma unroll 1
    for (int mu = 0; mu < 4; ++mu) {
      int cm = cc[0], sm = st[0], Lm = g.L[0];
      if (mu == 1) { cm = cc[1]; sm = st[1]; Lm = g.L[1]; }
      if (mu == 2) { cm = cc[2]; sm = st[2]; Lm = g.L[2]; }
      if (mu == 3) { cm = cc[3]; sm = st[3]; Lm = g.L[3]; }
      const int dn = cm == 0 ? x + (Lm - 1) * sm : x - sm;
      Cx<R> p[12], t[2][3];
      __syncwarp();
      gather_spinors<R>(in, cm + 1 == Lm ? x - cm * sm : x + sm, lane, sp);
      gather_links<R>(U, x, mu, lane, lk);
      __syncwarp();
      read_spinor<R>(sp, lane, p);
      hop_fwd_dispatch<R>(mu, p, lk + lane * 9, t);
      __syncwarp();
      gather_spinors<R>(in, dn, lane, sp);
      gather_links<R>(U, dn, mu, lane, lk);
      __syncwarp();
      read_spinor<R>(sp, lane, p);
      hop_bwd_dispatch<R>(mu, p, lk + lane * 9, t, acc);
    }
  }
  // own spinor for the diagonal, then (optionally) b for the epilogue
  Cx<R> o[12];
  __syncwarp();
  gather_spinors<R>(in, x, lane, sp);
  __syncwarp();
  read_spinor<R>(sp, lane, o);
  if constexpr (sizeof(R) == 4) {
    const R h = (R)0.5;
#pragma unroll
    for (int i = 0; i < 12; ++i) {
      const Cx<R> v = mk(diag * o[i].re - h * acc[i].re, diag * o[i].im - h * acc[i].im);
      o[i] = mk(a * v.re, a * v.im);
    }
  } else {
    const R ad = a * diag, ah = (R)-0.5 * a;
#pragma unroll
    for (int i = 0; i < 12; ++i) o[i] = mk(fma(ah, acc[i].re, ad * o[i].re), fma(ah, acc[i].im, ad * o[i].im));
  }
  if (b != nullptr) {
    Cx<R> bb[12];
    __syncwarp();
    gather_spinors<R>(b, x, lane, sp);
    __syncwarp();
    read_spinor<R>(sp, lane, bb);
#pragma unroll
    for (int i = 0; i < 12; ++i) o[i] = mk(o[i].re + c * bb[i].re, o[i].im + c * bb[i].im);
  }
  // coalesced store through the staging buffer: consecutive lanes write consecutive pieces
  __syncwarp();
  {
    typename S::V *q = sp + lane * S::STRIDE;
    if (sizeof(R) == 4) {
#pragma unroll
      for (int i = 0; i < 6; ++i)
        reinterpret_cast<float4 *>(q)[i] =
            make_float4((float)o[2 * i].re, (float)o[2 * i].im, (float)o[2 * i + 1].re, (float)o[2 * i + 1].im);
    } else {
#pragma unroll
      for (int i = 0; i < 12; ++i) reinterpret_cast<double2 *>(q)[i] = make_double2((double)o[i].re, (double)o[i].im);
    }
  }
  __syncwarp();
  typename S::V *dst = reinterpret_cast<typename S::V *>(out);
#pragma unroll
  for (int k = 0; k < S::PIECES; ++k) {
    const int cidx = lane + 32 * k, i = cidx / S::PIECES, j = cidx - i * S::PIECES;
    if (warp_first + i < V) dst[(long long)(warp_first + i) * S::PIECES + j] = sp[i * S::STRIDE + j];
  }
}

// ---------------------------------------------------------------------------
// Tiled FP32 apply, for extents divisible by 8 x 2 x 2 x 2: a warp owns one such tile, a lane the
// two sites of one (x0, x1, x2) that differ in x3. What bounded the one-site-per-thread form was
// the L1 path (91 % busy): 36 strided 8-byte link loads per site, each touching 32 sectors, and
// half spinors exchanged through shared memory behind block barriers. Here
//  * the tile's links and the links of its backward faces are copied into shared memory once by
//    coalesced 16-byte asynchronous copies and serve every vector of a batch (records of 304 B and
//    80 B: conflict-free 16-byte reads);
//  * spinors are read in 32-byte pieces, one sector each;
//  * a direction's two hops need the projected spinor of x + mu and U_{x-mu}^dagger times that of
//    x - mu. Each lane projects its own spinor for both, and the lanes of a row rotate them: the
//    first lane sends the forward half spinor of the site beyond the last one, the last lane the
//    backward product of the site before the first one, so every lane does two link products per
//    direction and no work for a neighbour is done twice inside the tile;
//  * the two x3 neighbours inside the tile are in one lane: no exchange at all.
// A warp waits for no other warp. Two sites per lane (about 255 registers, 8 warps per SM) give each
// warp twice the loads in flight, and a direction's outside spinors are requested while the one
// before it is worked on: with so few warps the loads' latency is what bounds it (L1 path 40 % busy,
// issue slots 40 %). 32^3 x 64: 250 us (4.0 TB/s), the one-site form 353 us. 24 vectors on 16^3 x 32
// with the MR step (mr_step_batch_kernel): 528 us, before 836 us; without the early requests and with
// the sums met in a block reduction per vector 691 us; with the step applied while r is read (6
// vector passes, not 7) 677 us, the doubled face loads costing what the pass saves; 12 warps of 168
// registers sharing the staged links 718 us.
// ---------------------------------------------------------------------------

template <bool A32>
__device__ __forceinline__ void load_spinor32(const Cx<float> *__restrict__ f, int x, Cx<float> (&p)[12]) {
  const float *q = reinterpret_cast<const float *>(f) + (long long)x * 24;
  float v[24];
  if (A32) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
      asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
          : "=f"(v[8 * i]), "=f"(v[8 * i + 1]), "=f"(v[8 * i + 2]), "=f"(v[8 * i + 3]), "=f"(v[8 * i + 4]),
            "=f"(v[8 * i + 5]), "=f"(v[8 * i + 6]), "=f"(v[8 * i + 7])
          : "l"(q + 8 * i));
  } else {
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      const float4 w = __ldg(reinterpret_cast<const float4 *>(q) + i);
      v[4 * i] = w.x;
      v[4 * i + 1] = w.y;
      v[4 * i + 2] = w.z;
      v[4 * i + 3] = w.w;
    }
  }
#pragma unroll
  for (int i = 0; i < 12; ++i) p[i] = mk(v[2 * i], v[2 * i + 1]);
}

template <bool A32>
__device__ __forceinline__ void store_spinor32(Cx<float> *f, int x, const Cx<float> (&p)[12]) {
  float *q = reinterpret_cast<float *>(f) + (long long)x * 24;
  if (A32) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
      asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(q + 8 * i), "f"(p[4 * i].re),
                   "f"(p[4 * i].im), "f"(p[4 * i + 1].re), "f"(p[4 * i + 1].im), "f"(p[4 * i + 2].re),
                   "f"(p[4 * i + 2].im), "f"(p[4 * i + 3].re), "f"(p[4 * i + 3].im)
                   : "memory");
  } else {
#pragma unroll
    for (int i = 0; i < 6; ++i)
      reinterpret_cast<float4 *>(q)[i] = make_float4(p[2 * i].re, p[2 * i].im, p[2 * i + 1].re, p[2 * i + 1].im);
  }
}

// t = U h (DAG false) or U^dagger h, for both spin rows of h
template <bool DAG>
__device__ __forceinline__ void link_times4(const Cx<float> (&u)[9], const Cx<float> (&h)[6], Cx<float> (&t)[6]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    Cx<float> t0 = mk(0.f, 0.f), t1 = mk(0.f, 0.f);
#pragma unroll
    for (int bb = 0; bb < 3; ++bb) {
      if (DAG) {
        cmac_conj(t0, u[bb * 3 + a], h[bb]);
        cmac_conj(t1, u[bb * 3 + a], h[3 + bb]);
      } else {
        cmac(t0, u[a * 3 + bb], h[bb]);
        cmac(t1, u[a * 3 + bb], h[3 + bb]);
      }
    }
    t[a] = t0;
    t[3 + a] = t1;
  }
}

// acc_up += t, acc_dn -= A_mu^dagger t (forward hop) or += (backward hop)
template <int MU, bool FWD>
__device__ __forceinline__ void reconstruct4(const Cx<float> (&t)[6], Cx<float> (&acc)[12]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    Cx<float> l0, l1;
    adag_times<float, MU>(t[c], t[3 + c], l0, l1);
    acc[c] = acc[c] + t[c];
    acc[3 + c] = acc[3 + c] + t[3 + c];
    if (FWD) {
      acc[6 + c] = acc[6 + c] - l0;
      acc[9 + c] = acc[9 + c] - l1;
    } else {
      acc[6 + c] = acc[6 + c] + l0;
      acc[9 + c] = acc[9 + c] + l1;
    }
  }
}

namespace {

// staged links, in 16-byte units: a site's four links (288 B, padded), and one link of a face site
// as the 80 bytes around it that start on a 16-byte boundary. U16: the links start on 16 bytes; else (on an odd 8) a
// record begins 8 bytes before its site, so that it too is copied in whole units, and fills its padding.
constexpr int kRec = 19, kHalo = 5;
constexpr int kHaloX = 0, kHaloY = 8, kHaloZ = 40, kHaloT = 72, kHaloSites = 104;
constexpr int kTiles = 4;      // tiles of a CTA
constexpr int kMaxChunk = 32;  // vectors of a CTA
constexpr int kTileUnits = 64 * kRec + kHaloSites * kHalo;
constexpr size_t kPairSmem = (size_t)kTiles * kTileUnits * 16;

// first 16-byte unit of link mu in a record; every second link starts 8 bytes into it
template <bool U16>
__host__ __device__ constexpr int link_unit(int mu) { return (72 * mu + (U16 ? 0 : 8)) / 16; }

// one unit of the links, which lie in [U, end): the units of links on an odd 8 bytes that reach over either end are
// copied by the half that is inside
template <bool U16>
__device__ __forceinline__ void copy16(float4 *dst, const char *src, const char *U, const char *end) {
  const unsigned int d = (unsigned int)__cvta_generic_to_shared(dst);
  if (!U16 && src < U)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d + 8), "l"(src + 8) : "memory");
  else if (!U16 && src + 16 > end)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
  else
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}

template <int MU, bool U16>
__device__ __forceinline__ void staged_link(const float4 *q, Cx<float> (&u)[9]) {
  if ((MU % 2 == 0) == U16) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 w = q[i];
      u[2 * i] = mk(w.x, w.y);
      u[2 * i + 1] = mk(w.z, w.w);
    }
    const float2 w = *reinterpret_cast<const float2 *>(q + 4);
    u[8] = mk(w.x, w.y);
  } else {
    const float2 w = reinterpret_cast<const float2 *>(q)[1];
    u[0] = mk(w.x, w.y);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 v = q[1 + i];
      u[1 + 2 * i] = mk(v.x, v.y);
      u[2 + 2 * i] = mk(v.z, v.w);
    }
  }
}

__device__ __forceinline__ void rotate6(const Cx<float> (&s)[6], int src, Cx<float> (&d)[6]) {
#pragma unroll
  for (int i = 0; i < 6; ++i)
    d[i] = mk(__shfl_sync(0xffffffffu, s[i].re, src), __shfl_sync(0xffffffffu, s[i].im, src));
}

// the two hops of direction MU (0, 1, 2) for the lane's site with spinor p: q is the spinor of the site
// beyond the row that the lane read (first lane: the one after the last, last lane: the one before
// the first; others none), fsrc / bsrc the lanes holding x + mu and x - mu (cyclic in the row), own /
// face the staged links of the site and of the site before the first one
template <int MU, bool U16>
__device__ __forceinline__ void row_hops(const Cx<float> (&p)[12], const Cx<float> (&q)[12], bool first, bool last,
                                         int fsrc, int bsrc, const float4 *own, const float4 *face,
                                         Cx<float> (&acc)[12]) {
  Cx<float> e[6], h[6], t[6], u[9];
  // e = (1 - gamma) q on the first lane, (1 + gamma) q on the last: only the sign of A q_dn differs
  const float sg = first ? -1.f : 1.f;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    Cx<float> a0, a1;
    a_times<float, MU>(q[6 + c], q[9 + c], a0, a1);
    e[c] = mk(fmaf(sg, a0.re, q[c].re), fmaf(sg, a0.im, q[c].im));
    e[3 + c] = mk(fmaf(sg, a1.re, q[3 + c].re), fmaf(sg, a1.im, q[3 + c].im));
  }
  hop_project<float, MU, true>(p, h);
#pragma unroll
  for (int i = 0; i < 6; ++i) h[i] = mk(first ? e[i].re : h[i].re, first ? e[i].im : h[i].im);
  rotate6(h, fsrc, t);
  staged_link<MU, U16>(own + link_unit<U16>(MU), u);
  link_times4<false>(u, t, h);
  reconstruct4<MU, true>(h, acc);
  hop_project<float, MU, false>(p, h);
#pragma unroll
  for (int i = 0; i < 6; ++i) h[i] = mk(last ? e[i].re : h[i].re, last ? e[i].im : h[i].im);
  staged_link<MU, U16>(last ? face : own + link_unit<U16>(MU), u);
  link_times4<true>(u, h, t);
  rotate6(t, bsrc, h);
  reconstruct4<MU, false>(h, acc);
}

}  // namespace

// SUMS: also the step length of an MR iteration on each vector, omega <out, in> / |out|^2, from the
// values the kernel holds anyway: FP32 sums over a site and the 64 sites of a tile, FP64 over the CTA's tiles, the
// partials, the final sum and the quotient, into mr.alpha[v]
struct MrStep {
  double *partials;       // [vector][CTA][3]
  unsigned int *tickets;  // [vector], zero
  double omega;
  float2 *alpha;          // [vector], written by the last CTA of the vector
};

// out_v = a (D in_v) + c b_v for the vectors [chunk blockIdx.y, ...) of nvec (stride ldv complex)
template <bool A32, bool SHIFT, bool SUMS, bool U16>
__global__ void __launch_bounds__(32 * kTiles, 2)
    dslash4_pair_kernel(const Cx<float> *__restrict__ U, const Cx<float> *__restrict__ in, Cx<float> *__restrict__ out,
                        Geo4 g, float diag, const Cx<float> *__restrict__ b, float a, float c, long long ldv,
                        const double *__restrict__ shift, int nvec, int chunk, MrStep mr) {
  extern __shared__ float4 staged[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int l0 = lane & 7, l1 = (lane >> 3) & 1, l2 = lane >> 4;
  const int tiles = (int)(g.nsites / 64);
  const int tile = blockIdx.x * kTiles + w;
  const bool live = tile < tiles;  // whole warps
  const int s1 = g.L[0], s2 = s1 * g.L[1], s3 = s2 * g.L[2];
  int tb = live ? tile : 0;
  const int n0 = g.L[0] / 8, n1 = g.L[1] / 2, n2 = g.L[2] / 2;
  const int o0 = (tb % n0) * 8;
  tb /= n0;
  const int o1 = (tb % n1) * 2;
  tb /= n1;
  const int o2 = (tb % n2) * 2, o3 = (tb / n2) * 2;
  // coordinates just outside the tile, periodic
  const int p0 = o0 + 8 == g.L[0] ? 0 : o0 + 8, m0 = o0 == 0 ? g.L[0] - 1 : o0 - 1;
  const int p1 = o1 + 2 == g.L[1] ? 0 : o1 + 2, m1 = o1 == 0 ? g.L[1] - 1 : o1 - 1;
  const int p2 = o2 + 2 == g.L[2] ? 0 : o2 + 2, m2 = o2 == 0 ? g.L[2] - 1 : o2 - 1;
  const int p3 = o3 + 2 == g.L[3] ? 0 : o3 + 2, m3 = o3 == 0 ? g.L[3] - 1 : o3 - 1;
  float4 *rec = staged + w * kTileUnits, *halo = rec + 64 * kRec;
  if (live) {
    const char *U0 = reinterpret_cast<const char *>(U), *U1 = U0 + g.nsites * 288, *Ub = U16 ? U0 : U0 - 8;
    constexpr int n = U16 ? 18 : 19;  // units of a record
    const long long org = o0 + (long long)o1 * s1 + (long long)o2 * s2 + (long long)o3 * s3;
    // own links: 8 rows of 8 sites
#pragma unroll 4
    for (int it = 0; it < 2 * n; ++it) {
      const int idx = it * 32 + lane, row = idx / (8 * n), k = idx - row * 8 * n, site = k / n;
      const long long x = org + (row & 1) * s1 + ((row >> 1) & 1) * s2 + (row >> 2) * s3;
      copy16<U16>(rec + (row * 8 + site) * kRec + (k - site * n), Ub + x * 288 + k * 16 - (n - 18) * 16 * site, U0, U1);
    }
    // backward faces: 8 sites of the x0 face, 4 rows of 8 sites of each other face
#pragma unroll
    for (int it = 0; it < 2; ++it) {
      const int idx = it * 32 + lane, e = idx / kHalo, k = idx - e * kHalo;
      const long long x = org - o0 + m0 + (e & 1) * s1 + ((e >> 1) & 1) * s2 + (e >> 2) * s3;
      if (idx < 8 * kHalo) copy16<U16>(halo + idx, Ub + x * 288 + k * 16, U0, U1);
    }
#pragma unroll
    for (int mu = 1; mu < 4; ++mu) {
      const long long face = mu == 1 ? org + (long long)(m1 - o1) * s1
                                     : mu == 2 ? org + (long long)(m2 - o2) * s2 : org + (long long)(m3 - o3) * s3;
      const int sa = mu == 1 ? s2 : s1, sb = mu == 3 ? s2 : s3;
      const int h0 = (mu == 1 ? kHaloY : mu == 2 ? kHaloZ : kHaloT) * kHalo;
#pragma unroll
      for (int it = 0; it < 5; ++it) {
        const int idx = it * 32 + lane, row = idx / 40, e = (idx - row * 40) / kHalo, k = idx % kHalo;
        const long long x = face + (row & 1) * sa + (row >> 1) * sb + e;
        copy16<U16>(halo + h0 + idx, Ub + x * 288 + (link_unit<U16>(mu) + k) * 16, U0, U1);
      }
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  const int row12 = (o1 + l1) * s1 + (o2 + l2) * s2;
  const int xA = o0 + l0 + row12 + o3 * s3, xB = xA + s3;
  const float4 *recA = rec + lane * kRec, *recB = recA + 32 * kRec;
  // the outside site this lane reads for the rows along x0, x1 and x2 of site A (site B: + s3)
  const int dx = (l0 == 0 ? p0 - o0 : m0 - (o0 + 7));
  const int outX = xA + dx, outY = xA + (l1 == 0 ? p1 - o1 : m1 - (o1 + 1)) * s1,
            outZ = xA + (l2 == 0 ? p2 - o2 : m2 - (o2 + 1)) * s2;
  const int fX = (lane & 24) | ((l0 + 1) & 7), bX = (lane & 24) | ((l0 + 7) & 7);
  const float4 *hX = halo + (kHaloX + l1 + 2 * l2) * kHalo, *hY = halo + (kHaloY + l0 + 8 * l2) * kHalo,
               *hZ = halo + (kHaloZ + l0 + 8 * l1) * kHalo, *hT = halo + (kHaloT + lane) * kHalo;
  const int v0 = blockIdx.y * chunk, v1 = v0 + chunk < nvec ? v0 + chunk : nvec;
  in += v0 * ldv;
  out += v0 * ldv;
  if (b != nullptr) b += v0 * ldv;
  __shared__ float sh[SUMS ? kMaxChunk : 1][kTiles][3];  // a tile's sums
  for (int v = v0; v < v1; ++v) {
    const float dg = SHIFT ? diag + (float)shift[v] : diag;
    float sums[3] = {0.f, 0.f, 0.f};
    if (live) {
      Cx<float> pA[12], pB[12], aA[12], aB[12];
      load_spinor32<A32>(in, xA, pA);
      load_spinor32<A32>(in, xB, pB);
      Cx<float> qA[12], qB[12], nA[12], nB[12];
#pragma unroll
      for (int i = 0; i < 12; ++i) qA[i] = qB[i] = mk(0.f, 0.f);
      if (l0 == 0 || l0 == 7) {
        load_spinor32<A32>(in, outX, qA);
        load_spinor32<A32>(in, outX + s3, qB);
      }
#pragma unroll
      for (int i = 0; i < 12; ++i) aA[i] = aB[i] = mk(0.f, 0.f);
      // each direction's outside spinors are requested while the one before it is worked on
      load_spinor32<A32>(in, outY, nA);
      load_spinor32<A32>(in, outY + s3, nB);
      if (v == v0) {  // the links are on their way while the first spinors are
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
      }
      row_hops<0, U16>(pA, qA, l0 == 0, l0 == 7, fX, bX, recA, hX, aA);
      row_hops<0, U16>(pB, qB, l0 == 0, l0 == 7, fX, bX, recB, hX + 4 * kHalo, aB);
      load_spinor32<A32>(in, outZ, qA);
      row_hops<1, U16>(pA, nA, l1 == 0, l1 == 1, lane ^ 8, lane ^ 8, recA, hY, aA);
      load_spinor32<A32>(in, outZ + s3, qB);
      row_hops<1, U16>(pB, nB, l1 == 0, l1 == 1, lane ^ 8, lane ^ 8, recB, hY + 16 * kHalo, aB);
      load_spinor32<A32>(in, xA + (m3 - o3) * s3, nA);
      row_hops<2, U16>(pA, qA, l2 == 0, l2 == 1, lane ^ 16, lane ^ 16, recA, hZ, aA);
      load_spinor32<A32>(in, xA + (p3 - o3) * s3, nB);
      row_hops<2, U16>(pB, qB, l2 == 0, l2 == 1, lane ^ 16, lane ^ 16, recB, hZ + 16 * kHalo, aB);
      {  // direction 3: the neighbours inside the tile are the lane's own two sites
        Cx<float> h[6], t[6], t2[6], u[9];
        staged_link<3, U16>(recA + link_unit<U16>(3), u);
        hop_project<float, 3, true>(pB, h);
        link_times4<false>(u, h, t);
        reconstruct4<3, true>(t, aA);
        hop_project<float, 3, false>(pA, h);
        link_times4<true>(u, h, t);
        staged_link<3, U16>(hT, u);
        hop_project<float, 3, false>(nA, h);
        link_times4<true>(u, h, t2);
        reconstruct4<3, false>(t2, aA);
        staged_link<3, U16>(recB + link_unit<U16>(3), u);
        hop_project<float, 3, true>(nB, h);
        link_times4<false>(u, h, t2);
        reconstruct4<3, true>(t2, aB);
        reconstruct4<3, false>(t, aB);
      }
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        Cx<float>(&p)[12] = half ? pB : pA;
        Cx<float>(&acc)[12] = half ? aB : aA;
        const int x = half ? xB : xA;
        float site[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int i = 0; i < 12; ++i) {
          const Cx<float> o =
              mk(a * (dg * p[i].re - 0.5f * acc[i].re), a * (dg * p[i].im - 0.5f * acc[i].im));
          if (SUMS) {
            site[0] += o.re * p[i].re + o.im * p[i].im;
            site[1] += o.re * p[i].im - o.im * p[i].re;
            site[2] += o.re * o.re + o.im * o.im;
          }
          p[i] = o;
        }
        if (SUMS) {
#pragma unroll
          for (int k = 0; k < 3; ++k) sums[k] += site[k];
        }
        if (b != nullptr) {
          Cx<float> q[12];
          load_spinor32<A32>(b, x, q);
#pragma unroll
          for (int i = 0; i < 12; ++i) p[i] = mk(p[i].re + c * q[i].re, p[i].im + c * q[i].im);
        }
        store_spinor32<A32>(out, x, p);
      }
    }
    if (SUMS) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sums[k] += __shfl_xor_sync(0xffffffffu, sums[k], o);
        if (lane == 0) sh[v - v0][w][k] = sums[k];
      }
    }
    in += ldv;
    out += ldv;
    if (b != nullptr) b += ldv;
  }
  if (SUMS) {
    // the CTA's sums of every vector, then, in the last CTA of a vector, its FP64 sum over all CTAs
    __shared__ bool last[kMaxChunk];
    __syncthreads();
    const int j = threadIdx.x;
    if (j < v1 - v0) {
      const int v = v0 + j;
      double *part = mr.partials + (long long)v * gridDim.x * 3;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        double t = 0.0;
#pragma unroll
        for (int q = 0; q < kTiles; ++q) t += (double)sh[j][q][k];
        part[blockIdx.x * 3 + k] = t;
      }
      __threadfence();
      last[j] = atomicAdd(mr.tickets + v, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    __shared__ double shd[32 * 3];
    for (int i = 0; i < v1 - v0; ++i) {
      if (!last[i]) continue;
      const int v = v0 + i;
      const volatile double *part = mr.partials + (long long)v * gridDim.x * 3;
      __threadfence();
      double s[3] = {0.0, 0.0, 0.0};
      for (unsigned int q = threadIdx.x; q < gridDim.x; q += blockDim.x) {
#pragma unroll
        for (int k = 0; k < 3; ++k) s[k] += part[q * 3 + k];
      }
      block_sum<3>(s, shd);
      if (threadIdx.x == 0) {
        // a vanishing A r leaves r and x as they are
        mr.alpha[v] = s[2] > 0.0 ? make_float2((float)(mr.omega * s[0] / s[2]), (float)(mr.omega * s[1] / s[2]))
                                 : make_float2(0.f, 0.f);
        mr.tickets[v] = 0u;
      }
    }
  }
}

namespace {

// CTAs of one launch over the lattice, and the vectors each takes: the count that gives the least
// work on the busiest SM (2 CTAs resident on each of 152), staging the links counted as 0.6 vectors
int pair_ctas(const Geo4 &g) { return (int)((g.nsites / 64 + kTiles - 1) / kTiles); }
int pair_chunk(const Geo4 &g, int nvec) {
  int best = 1;
  double cost = 0.0;
  for (int c = 1; c <= nvec && c <= kMaxChunk; ++c) {
    const long long ctas = (long long)pair_ctas(g) * ((nvec + c - 1) / c);
    const double t = (double)((ctas + 303) / 304) * (c + 0.6);
    if (c == 1 || t < cost) {
      best = c;
      cost = t;
    }
  }
  return best;
}

template <bool A32, bool SHIFT, bool SUMS, bool U16 = true>
void launch_pair(const Cx<float> *U, const Cx<float> *in, Cx<float> *out, Geo4 g, double diag, const Cx<float> *b,
                 double a, double c, cudaStream_t s, int nvec, const double *shift, MrStep mr) {
  auto fn = dslash4_pair_kernel<A32, SHIFT, SUMS, U16>;
  MG_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPairSmem));
  const int chunk = pair_chunk(g, nvec);
  fn<<<dim3(pair_ctas(g), (nvec + chunk - 1) / chunk), 32 * kTiles, kPairSmem, s>>>(
      U, in, out, g, (float)diag, b, (float)a, (float)c, 12 * g.nsites, shift, nvec, chunk, mr);
  MG_LAUNCHED();
}

bool aligned(const void *p, uintptr_t n) { return (reinterpret_cast<uintptr_t>(p) & (n - 1)) == 0; }

// the tiled kernel takes lattices of whole 8 x 2 x 2 x 2 tiles; other shapes run the warp gather
bool pair_takes(const Geo4 &g) {
  return g.L[0] % 8 == 0 && g.L[1] % 2 == 0 && g.L[2] % 2 == 0 && g.L[3] % 2 == 0 &&
         std::getenv("MG_DSLASH4_GATHER") == nullptr;
}

}  // namespace

// true when the tiled kernel took the apply
static bool try_tile4(const Cx<float> *U, const Cx<float> *in, Cx<float> *out, Geo4 g, double diag,
                      const Cx<float> *b, double a, double c, cudaStream_t s, int nvec, const double *shift) {
  if (!pair_takes(g)) return false;
  const bool a32 = aligned(in, 32) && aligned(out, 32) && aligned(b, 32);
  auto run = [&](auto fn) { fn(U, in, out, g, diag, b, a, c, s, nvec, shift, MrStep{}); };
  // links on an odd 8 bytes come from a caller's own buffer (mg_dslash), never with shifts: their records begin 8
  // bytes before the site (32^3 x 64: 340 us; 8-byte copies 371, the warp gather 417, the tiled kernel before 355)
  if (!aligned(U, 16)) {
    if (shift != nullptr) return false;
    run(launch_pair<false, false, false, false>);
  } else if (a32)
    shift != nullptr ? run(launch_pair<true, true, false>) : run(launch_pair<true, false, false>);
  else
    shift != nullptr ? run(launch_pair<false, true, false>) : run(launch_pair<false, false, false>);
  return true;
}

bool launch_dslash4_mr(const Cx<float> *U, const Cx<float> *r, Cx<float> *Ar, Geo4 g, double diag, int nvec,
                       double omega, float2 *alpha, double *partials, long long partials_cap, unsigned int *tickets,
                       cudaStream_t s) {
  if (!pair_takes(g) || !aligned(U, 16) || (long long)pair_ctas(g) * 3 * nvec > partials_cap) return false;
  const MrStep mr{partials, tickets, omega, alpha};
  if (aligned(r, 32) && aligned(Ar, 32))
    launch_pair<true, false, true>(U, r, Ar, g, diag, nullptr, 1.0, 0.0, s, nvec, nullptr, mr);
  else
    launch_pair<false, false, true>(U, r, Ar, g, diag, nullptr, 1.0, 0.0, s, nvec, nullptr, mr);
  return true;
}

template <typename R>
void launch_dslash4(const Cx<R> *U, const Cx<R> *in, Cx<R> *out, Geo4 g, double diag, const Cx<R> *b, double a,
                    double c, cudaStream_t s, int nvec, const double *shift) {
  if constexpr (sizeof(R) == 4) {
    if (try_tile4(U, in, out, g, diag, b, a, c, s, nvec, shift)) return;
  }
  const int threads = 32 * DSLASH4_WARPS;
  const dim3 grid(grid_for(g.nsites, threads), nvec);
  if (shift != nullptr)
    dslash4_kernel<R, true><<<grid, threads, 0, s>>>(U, in, out, g, (R)diag, b, (R)a, (R)c, 12 * g.nsites, shift);
  else
    dslash4_kernel<R, false><<<grid, threads, 0, s>>>(U, in, out, g, (R)diag, b, (R)a, (R)c, 12 * g.nsites,
                                                      nullptr);
  MG_LAUNCHED();
}

template void launch_dslash4<double>(const Cx<double> *, const Cx<double> *, Cx<double> *, Geo4, double,
                                     const Cx<double> *, double, double, cudaStream_t, int, const double *);
template void launch_dslash4<float>(const Cx<float> *, const Cx<float> *, Cx<float> *, Geo4, double,
                                    const Cx<float> *, double, double, cudaStream_t, int, const double *);

}  // namespace mg
