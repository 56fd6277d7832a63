// Directional terms of the Wilson hopping operator (device functions).
//
//   H psi(x) = -1/2 sum_mu [ (1 - gamma_mu) U_mu(x) psi(x+mu)
//                          + (1 + gamma_mu) U_mu(x-mu)^dag psi(x-mu) ]
//
// (Wilson r = 1; the paper's operator D(U) of Eq. 1 with the clover term
// kept site-local.)  In the DeGrand-Rossi chiral basis every gamma_mu has the
// off-diagonal block form [[0, a_mu], [b_mu, 0]] with b_mu a_mu = 1:
//   a_x = i sigma_1, a_y = -i sigma_2, a_z = i sigma_3, a_t = 1,
//   b_x = -i sigma_1, b_y = i sigma_2, b_z = -i sigma_3, b_t = 1.
// Hence (1 -/+ gamma_mu) psi = [h ; -/+ b_mu h] with h = psi_up -/+ a_mu psi_dn,
// so each term needs one 2-spin half spinor, two SU(3) mat-vecs and a
// reconstruction with permutations and factors of +-1, +-i only.
// The -1/2 is applied by the caller.  Fermions are antiperiodic in t.
#pragma once
#include "common.cuh"

namespace mg {

// (a_mu d)[0], (a_mu d)[1] for a lower-spin pair d0 = psi_2, d1 = psi_3
template <int MU, typename T>
__device__ __forceinline__ void mul_a(cx<T> d0, cx<T> d1, cx<T>& o0, cx<T>& o1) {
  if (MU == 0) { o0 = times_i(d1); o1 = times_i(d0); }
  if (MU == 1) { o0 = -d1; o1 = d0; }
  if (MU == 2) { o0 = times_i(d0); o1 = -times_i(d1); }
  if (MU == 3) { o0 = d0; o1 = d1; }
}

// (b_mu g)[0], (b_mu g)[1]
template <int MU, typename T>
__device__ __forceinline__ void mul_b(cx<T> g0, cx<T> g1, cx<T>& o0, cx<T>& o1) {
  if (MU == 0) { o0 = -times_i(g1); o1 = -times_i(g0); }
  if (MU == 1) { o0 = g1; o1 = -g0; }
  if (MU == 2) { o0 = -times_i(g0); o1 = times_i(g1); }
  if (MU == 3) { o0 = g0; o1 = g1; }
}

// Neighbour of site c in direction MU (FWD: +mu, else -mu): its checkerboard
// index and the boundary sign (-1 when the hop crosses the t boundary with
// antiperiodic fermions).
template <int MU, bool FWD>
__device__ __forceinline__ int neighbour(const Geom& g, const int c[4], int& sgn) {
  int n[4] = {c[0], c[1], c[2], c[3]};
  sgn = 1;
  if (FWD) {
    n[MU] = (c[MU] + 1 == g.L[MU]) ? 0 : c[MU] + 1;
    if (MU == 3 && g.apbc && c[3] == g.L[3] - 1) sgn = -1;
  } else {
    n[MU] = (c[MU] == 0) ? g.L[MU] - 1 : c[MU] - 1;
    if (MU == 3 && g.apbc && c[3] == 0) sgn = -1;
  }
  return cb_index(g, n);
}

// The arithmetic of one hop term: acc += (1 -/+ gamma_mu) U psi for the
// neighbour spinor psi and the link u (U_mu(x) for FWD, U_mu(x - mu) to be
// used daggered otherwise), s = boundary sign x hopping weight.
template <typename T, int MU, bool FWD>
__device__ __forceinline__ void hop_apply(const cx<T> psi[12], const cx<T> u[9], T s, cx<T> acc[12]) {
  cx<T> h0[3], h1[3];
#pragma unroll
  for (int col = 0; col < 3; col++) {
    cx<T> a0, a1;
    mul_a<MU, T>(psi[6 + col], psi[9 + col], a0, a1);
    if (FWD) {
      h0[col] = psi[col] - a0;
      h1[col] = psi[3 + col] - a1;
    } else {
      h0[col] = psi[col] + a0;
      h1[col] = psi[3 + col] + a1;
    }
  }
  if (sizeof(T) == 4 || s != (T)1) {   // in FP64 the twelve products are 9 % of a hop: only where the sign or a weight asks
#pragma unroll
    for (int col = 0; col < 3; col++) {
      h0[col] = s * h0[col];
      h1[col] = s * h1[col];
    }
  }
  cx<T> g0[3], g1[3];
#pragma unroll
  for (int a = 0; a < 3; a++) {
    g0[a] = mkc<T>(0, 0);
    g1[a] = mkc<T>(0, 0);
#pragma unroll
    for (int b = 0; b < 3; b++) {
      if (FWD) {
        g0[a] = cfma(u[a * 3 + b], h0[b], g0[a]);
        g1[a] = cfma(u[a * 3 + b], h1[b], g1[a]);
      } else {
        g0[a] = cfma_conj(u[b * 3 + a], h0[b], g0[a]);
        g1[a] = cfma_conj(u[b * 3 + a], h1[b], g1[a]);
      }
    }
  }
#pragma unroll
  for (int col = 0; col < 3; col++) {
    acc[col] = acc[col] + g0[col];
    acc[3 + col] = acc[3 + col] + g1[col];
    cx<T> b0, b1;
    mul_b<MU, T>(g0[col], g1[col], b0, b1);
    if (FWD) {
      acc[6 + col] = acc[6 + col] - b0;
      acc[9 + col] = acc[9 + col] - b1;
    } else {
      acc[6 + col] = acc[6 + col] + b0;
      acc[9 + col] = acc[9 + col] + b1;
    }
  }
}

// acc += (1 -/+ gamma_mu) U psi(neighbour), without the -1/2.
//  in:    spinor half of parity 1-par (the neighbours' parity)
//  gauge: full internal gauge field
//  par,i,c: parity, checkerboard index and coordinates of the output site
template <typename T, int MU, bool FWD>
__device__ __forceinline__ void hop_term(const Geom& g, const T* __restrict__ in, const T* __restrict__ gauge,
                                         int par, int i, const int c[4], cx<T> acc[12]) {
  int sgn;
  const int j = neighbour<MU, FWD>(g, c, sgn);
  cx<T> psi[12];
  SpinorIO<T>::load(in, g.Vh, j, psi);
  cx<T> u[9];
  if (FWD)
    load_link<T>(gauge, g.Vh, par, MU, i, u);      // U_mu(x)
  else
    load_link<T>(gauge, g.Vh, 1 - par, MU, j, u);  // U_mu(x - mu)
  hop_apply<T, MU, FWD>(psi, u, (T)sgn * (T)g.w[MU], acc);   // boundary sign and the direction's hopping weight
}

// Sum of the hop terms selected by `dirmask` (bit d: d < 4 forward mu = d,
// d >= 4 backward mu = d - 4), without the -1/2.
template <typename T>
__device__ __forceinline__ void hop_sum(const Geom& g, const T* __restrict__ in, const T* __restrict__ gauge,
                                        int par, int i, const int c[4], int dirmask, cx<T> acc[12]) {
  if (dirmask & 0x01) hop_term<T, 0, true>(g, in, gauge, par, i, c, acc);
  if (dirmask & 0x10) hop_term<T, 0, false>(g, in, gauge, par, i, c, acc);
  if (dirmask & 0x02) hop_term<T, 1, true>(g, in, gauge, par, i, c, acc);
  if (dirmask & 0x20) hop_term<T, 1, false>(g, in, gauge, par, i, c, acc);
  if (dirmask & 0x04) hop_term<T, 2, true>(g, in, gauge, par, i, c, acc);
  if (dirmask & 0x40) hop_term<T, 2, false>(g, in, gauge, par, i, c, acc);
  if (dirmask & 0x08) hop_term<T, 3, true>(g, in, gauge, par, i, c, acc);
  if (dirmask & 0x80) hop_term<T, 3, false>(g, in, gauge, par, i, c, acc);
}

// Multi-RHS form of hop_term: the link is loaded once and applied to the
// neighbour spinors of nr <= NR right-hand sides (in + r * stride).
template <typename T, int MU, bool FWD, int NR>
__device__ __forceinline__ void hop_term_nr(const Geom& g, const T* __restrict__ in, size_t stride, int nr,
                                            const T* __restrict__ gauge, int par, int i, const int c[4],
                                            cx<T> acc[NR][12]) {
  int sgn;
  const int j = neighbour<MU, FWD>(g, c, sgn);
  cx<T> u[9];
  if (FWD)
    load_link<T>(gauge, g.Vh, par, MU, i, u);
  else
    load_link<T>(gauge, g.Vh, 1 - par, MU, j, u);
  const T s = (T)sgn * (T)g.w[MU];   // boundary sign and the direction's hopping weight
#pragma unroll
  for (int r = 0; r < NR; r++) {
    if (r >= nr) break;
    cx<T> psi[12];
    SpinorIO<T>::load(in + r * stride, g.Vh, j, psi);
    cx<T> h0[3], h1[3];
#pragma unroll
    for (int col = 0; col < 3; col++) {
      cx<T> a0, a1;
      mul_a<MU, T>(psi[6 + col], psi[9 + col], a0, a1);
      if (FWD) {
        h0[col] = s * (psi[col] - a0);
        h1[col] = s * (psi[3 + col] - a1);
      } else {
        h0[col] = s * (psi[col] + a0);
        h1[col] = s * (psi[3 + col] + a1);
      }
    }
#pragma unroll
    for (int a = 0; a < 3; a++) {
      cx<T> g0 = mkc<T>(0, 0), g1 = mkc<T>(0, 0);
#pragma unroll
      for (int b = 0; b < 3; b++) {
        if (FWD) {
          g0 = cfma(u[a * 3 + b], h0[b], g0);
          g1 = cfma(u[a * 3 + b], h1[b], g1);
        } else {
          g0 = cfma_conj(u[b * 3 + a], h0[b], g0);
          g1 = cfma_conj(u[b * 3 + a], h1[b], g1);
        }
      }
      acc[r][a] = acc[r][a] + g0;
      acc[r][3 + a] = acc[r][3 + a] + g1;
      cx<T> b0, b1;
      mul_b<MU, T>(g0, g1, b0, b1);
      if (FWD) {
        acc[r][6 + a] = acc[r][6 + a] - b0;
        acc[r][9 + a] = acc[r][9 + a] - b1;
      } else {
        acc[r][6 + a] = acc[r][6 + a] + b0;
        acc[r][9 + a] = acc[r][9 + a] + b1;
      }
    }
  }
}

template <typename T, int NR>
__device__ __forceinline__ void hop_sum_nr(const Geom& g, const T* __restrict__ in, size_t stride, int nr,
                                           const T* __restrict__ gauge, int par, int i, const int c[4], int dirmask,
                                           cx<T> acc[NR][12]) {
  if (dirmask & 0x01) hop_term_nr<T, 0, true, NR>(g, in, stride, nr, gauge, par, i, c, acc);
  if (dirmask & 0x10) hop_term_nr<T, 0, false, NR>(g, in, stride, nr, gauge, par, i, c, acc);
  if (dirmask & 0x02) hop_term_nr<T, 1, true, NR>(g, in, stride, nr, gauge, par, i, c, acc);
  if (dirmask & 0x20) hop_term_nr<T, 1, false, NR>(g, in, stride, nr, gauge, par, i, c, acc);
  if (dirmask & 0x04) hop_term_nr<T, 2, true, NR>(g, in, stride, nr, gauge, par, i, c, acc);
  if (dirmask & 0x40) hop_term_nr<T, 2, false, NR>(g, in, stride, nr, gauge, par, i, c, acc);
  if (dirmask & 0x08) hop_term_nr<T, 3, true, NR>(g, in, stride, nr, gauge, par, i, c, acc);
  if (dirmask & 0x80) hop_term_nr<T, 3, false, NR>(g, in, stride, nr, gauge, par, i, c, acc);
}

// out = C x for a packed two-block clover (A or A^{-1}) at site i.
template <typename T>
__device__ __forceinline__ void clover_mul(const T* __restrict__ clov, int Vh, int i, const cx<T> x[12], cx<T> y[12]) {
#pragma unroll
  for (int b = 0; b < 2; b++) {
    T r[36];
    CloverIO<T>::load_block(clov, Vh, i, b, r);
    herm6_apply<T>(r, x + 6 * b, y + 6 * b);
  }
}

// --------------------------------------------------------------------------- four lanes per site
// The hop sum and the clover product with a site's work spread over four
// neighbouring lanes, for lattices that do not fill the GPU with one site per
// thread: lane (k, b) = (l & 1, l >> 1) applies half-spinor component k of the
// forward (b = 0) or backward (b = 1) hop of every dimension -- a quarter of
// the arithmetic, with no divergence: what depends on the lane is which
// addresses are read and a few signs -- and ends with the three colours of spin
// 2 b + k.  An FP64 instruction of a warp occupies its scheduler's FP64 unit
// for 64 cycles on GB300, so a site per thread is a chain of about 1300 x 64
// cycles however many SMs are idle.
template <typename T>
__device__ __forceinline__ T flip(T v, bool neg);
template <>
__device__ __forceinline__ float flip<float>(float v, bool neg) {
  return __int_as_float(__float_as_int(v) ^ (neg ? (int)0x80000000 : 0));
}
template <>
__device__ __forceinline__ double flip<double>(double v, bool neg) {
  return __hiloint2double(__double2hiint(v) ^ (neg ? (int)0x80000000 : 0), __double2loint(v));
}

// one dimension: adds the lane's g to its upper sum and (+- b_mu) g to the lower spin it reaches
template <typename T, int MU>
__device__ __forceinline__ void lane_hop(const Geom& g, const T* __restrict__ in, const T* __restrict__ gauge, int par,
                                         int i, const int c[4], int k, int b, cx<T> up[3], cx<T> lo[2][3]) {
  using V2 = typename std::conditional<sizeof(T) == 4, float2, double2>::type;
  int sf, sb;
  const int jf = neighbour<MU, true>(g, c, sf), jb = neighbour<MU, false>(g, c, sb);
  const int j = b ? jb : jf, sgn = b ? sb : sf;
  // link entry (r, q) of U (forward) or U^dag (backward: transposed address, conjugated)
  const V2* u = reinterpret_cast<const V2*>(gauge) + (size_t)((b ? 1 - par : par) * 4 + MU) * 9 * g.Vh + (b ? j : i);
  const size_t sr = (size_t)(b ? 1 : 3) * g.Vh, sq = (size_t)(b ? 3 : 1) * g.Vh;
  V2 l[9];
#pragma unroll
  for (int r = 0; r < 3; r++)
#pragma unroll
    for (int q = 0; q < 3; q++) l[3 * r + q] = u[r * sr + q * sq];
  // h = psi_k -+ (a_mu psi_dn)_k: a_x = i s1, a_y = -i s2, a_z = i s3, a_t = 1
  const int dn = MU < 2 ? 3 - k : 2 + k;
  cx<T> h[3];
#pragma unroll
  for (int col = 0; col < 3; col++) {
    const cx<T> x = SpinorIO<T>::get(in, g.Vh, j, 3 * k + col), d = SpinorIO<T>::get(in, g.Vh, j, 3 * dn + col);
    cx<T> a;
    if (MU == 0) a = times_i(d);
    if (MU == 1) a = mkc(flip(d.re, k == 0), flip(d.im, k == 0));
    if (MU == 2) a = mkc(flip(d.im, k == 0), flip(d.re, k == 1));   // i d for k = 0, -i d for k = 1
    if (MU == 3) a = d;
    h[col] = mkc(x.re + flip(a.re, b == 0), x.im + flip(a.im, b == 0));
  }
  const T s = (T)sgn * (T)g.w[MU];
  if (s != (T)1) {
#pragma unroll
    for (int col = 0; col < 3; col++) h[col] = s * h[col];
  }
#pragma unroll
  for (int r = 0; r < 3; r++) {
    cx<T> v = mkc<T>(0, 0);
#pragma unroll
    for (int q = 0; q < 3; q++) v = cfma(mkc(l[3 * r + q].x, flip(l[3 * r + q].y, b == 1)), h[q], v);
    up[r] = up[r] + v;
    // lower spins: -+ b_mu g, b_x = -i s1, b_y = i s2, b_z = -i s3, b_t = 1 (minus for the forward hop)
    cx<T> w;
    if (MU == 0) w = mkc(v.im, -v.re);                                  // -i g_k onto spin 3 - k
    if (MU == 1) w = mkc(flip(v.re, k == 0), flip(v.im, k == 0));       // (b g)_0 = g_1, (b g)_1 = -g_0
    if (MU == 2) w = mkc(flip(v.im, k == 1), flip(v.re, k == 0));       // -i g_0, i g_1
    if (MU == 3) w = v;
    w = mkc(flip(w.re, b == 0), flip(w.im, b == 0));
    cx<T>& t = lo[MU < 2 ? 0 : 1][r];   // [0]: onto spin 3 - k, [1]: onto spin 2 + k
    t = t + w;
  }
}

// the hop sum of site i (without the -1/2): spin 2 b + k on lane (k, b); all
// lanes of the warp call it (lanes of a site past the end repeat another one)
template <typename T>
__device__ __forceinline__ void lane_hop_sum(const Geom& g, const T* __restrict__ in, const T* __restrict__ gauge,
                                             int par, int i, int k, int b, cx<T> acc[3]) {
  int c[4];
  cb_coords(g, i, par, c);
  cx<T> up[3], lo[2][3];
#pragma unroll
  for (int r = 0; r < 3; r++) up[r] = lo[0][r] = lo[1][r] = mkc<T>(0, 0);
  lane_hop<T, 0>(g, in, gauge, par, i, c, k, b, up, lo);
  lane_hop<T, 1>(g, in, gauge, par, i, c, k, b, up, lo);
  lane_hop<T, 2>(g, in, gauge, par, i, c, k, b, up, lo);
  lane_hop<T, 3>(g, in, gauge, par, i, c, k, b, up, lo);
  const unsigned full = 0xffffffffu;
  // forward and backward: the upper spin goes to lane b = 0, the lower ones to b = 1
#pragma unroll
  for (int r = 0; r < 3; r++) {
    const cx<T> s0 = b ? up[r] : lo[0][r], s1 = lo[1][r];
    const T r0 = __shfl_xor_sync(full, s0.re, 2), r1 = __shfl_xor_sync(full, s0.im, 2);
    const T r2 = __shfl_xor_sync(full, s1.re, 2), r3 = __shfl_xor_sync(full, s1.im, 2);
    if (b) {
      lo[0][r] = lo[0][r] + mkc(r0, r1);
      lo[1][r] = lo[1][r] + mkc(r2, r3);
    } else {
      up[r] = up[r] + mkc(r0, r1);
    }
  }
  // lanes b = 1: lo[1] is this lane's spin 2 + k, lo[0] belongs to the partner's
#pragma unroll
  for (int r = 0; r < 3; r++) {
    const T r0 = __shfl_xor_sync(full, lo[0][r].re, 1), r1 = __shfl_xor_sync(full, lo[0][r].im, 1);
    acc[r] = b ? lo[1][r] + mkc(r0, r1) : up[r];
  }
}

// rows 3 (s & 1) .. + 2 of the chiral block of spin s: y = C x, x = the lane's
// three components (its partner's come by shuffle).  The block is
// [[D0, B^dag], [B, D1]]: a lane reads its own Hermitian 3x3 block and B,
// transposed and conjugated on the upper rows.
template <typename T>
__device__ __forceinline__ void lane_clover(const T* __restrict__ clov, int Vh, int i, int k, int b, const cx<T> x[3],
                                            cx<T> y[3]) {
  using V2 = typename std::conditional<sizeof(T) == 4, float2, double2>::type;
  const unsigned full = 0xffffffffu;
  cx<T> z[3];
#pragma unroll
  for (int r = 0; r < 3; r++)
    z[r] = mkc(__shfl_xor_sync(full, x[r].re, 1), __shfl_xor_sync(full, x[r].im, 1));
  // real q of the block: FP32 in chunk q / 4 of four, FP64 in pair q / 2
  auto at = [&](int q) {
    if (sizeof(T) == 4)
      return reinterpret_cast<const T*>(clov) + ((size_t)(9 * b + q / 4) * Vh + i) * 4 + q % 4;
    return reinterpret_cast<const T*>(clov) + ((size_t)(18 * b + q / 2) * Vh + i) * 2 + q % 2;
  };
  auto entry = [&](int m) {
    const V2 v = *reinterpret_cast<const V2*>(at(6 + 2 * m));
    return mkc(v.x, v.y);
  };
#pragma unroll
  for (int r = 0; r < 3; r++) {
    const T d = *at(3 * k + r);
    y[r] = mkc(d * x[r].re, d * x[r].im);
  }
  const cx<T> e10 = entry(k ? 9 : 0), e20 = entry(k ? 13 : 1), e21 = entry(k ? 14 : 2);
  y[1] = cfma(e10, x[0], y[1]);
  y[0] = cfma_conj(e10, x[1], y[0]);
  y[2] = cfma(e20, x[0], y[2]);
  y[0] = cfma_conj(e20, x[2], y[0]);
  y[2] = cfma(e21, x[1], y[2]);
  y[1] = cfma_conj(e21, x[2], y[1]);
  // B_{rq} = entry(3 + r, q) = packed index 3, 4, 5 | 6, 7, 8 | 10, 11, 12
#pragma unroll
  for (int r = 0; r < 3; r++)
#pragma unroll
    for (int q = 0; q < 3; q++) {
      const int mrq = (r == 2 ? 10 : 3 + 3 * r) + q, mqr = (q == 2 ? 10 : 3 + 3 * q) + r;
      const cx<T> e = entry(k ? mrq : mqr);
      y[r] = cfma(mkc(e.re, flip(e.im, k == 0)), z[q], y[r]);
    }
}

}  // namespace mg
