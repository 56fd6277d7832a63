// Fine-level Wilson-clover kernels for sm_103a.
//
//  * ABI <-> internal packing of spinors and gauge links
//  * clover construction A = (4+m0) + csw (i/4) sum_{mu!=nu} sigma_{mu nu} F_{mu nu}; anisotropic
//    reading: (sum_mu w_mu + m0) + (i/4) sum_{mu!=nu} c_{mu nu} sigma F with the hopping weights w_mu of the
//    directions and c = csw_t (planes containing t) or csw_s (spatial planes)
//    and its site inverse (FP64), the D_ee / D_oo of the paper's even-odd
//    split ("Red-black preconditioning": D_ee, D_oo are site-diagonal)
//  * the fused hopping kernel ("dslash") with clover / axpy epilogues, from
//    which D, D_p = 1 + H A^{-1}, D_r = 1 - H_eo A_o^{-1} H_oe A_e^{-1} and
//    b_r = b_e - H_eo A_o^{-1} b_o are composed
//  * the eight directional hopping terms (Galerkin coarse-link construction)
//  * Philox4x32-10 Gaussian start vectors of the null-vector setup
//
// One thread per lattice site; spinors, links and clover are read as
// 16-byte (float4 / double2) or 8-byte chunks in structure-of-chunks order so
// that a warp reads contiguous 512-byte spans.
#include <atomic>
#include <cmath>
#include <cstdio>
#include <algorithm>
#include <type_traits>
#include <vector>

#include "dfloat.cuh"
#include "internal.h"
#include "philox.cuh"
#include "wilson_dev.cuh"

namespace mg {

// --------------------------------------------------------------------------- sigma blocks
// sigma_{mu nu} = (i/2)[gamma_mu, gamma_nu] in the DeGrand-Rossi basis is
// block diagonal in chirality; c_sigma[plane][block][s][t] holds the 2x2
// blocks for the planes (01, 02, 03, 12, 13, 23).
__constant__ double c_sigma[6][2][2][2][2];

namespace {
struct HC {
  double re, im;
};
HC hmul(HC a, HC b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }

// Uploads the table to the current device (every clover build: 384 bytes).
void upload_sigma() {
  // gamma_mu as 4x4 complex, rows of the DeGrand-Rossi table
  HC G[4][4][4] = {};
  auto set = [&](int mu, int r, int col, double re, double im) { G[mu][r][col] = {re, im}; };
  set(0, 0, 3, 0, 1); set(0, 1, 2, 0, 1); set(0, 2, 1, 0, -1); set(0, 3, 0, 0, -1);   // gamma_x
  set(1, 0, 3, -1, 0); set(1, 1, 2, 1, 0); set(1, 2, 1, 1, 0); set(1, 3, 0, -1, 0);   // gamma_y
  set(2, 0, 2, 0, 1); set(2, 1, 3, 0, -1); set(2, 2, 0, 0, -1); set(2, 3, 1, 0, 1);   // gamma_z
  set(3, 0, 2, 1, 0); set(3, 1, 3, 1, 0); set(3, 2, 0, 1, 0); set(3, 3, 1, 1, 0);     // gamma_t
  double host[6][2][2][2][2];
  int plane = 0;
  for (int mu = 0; mu < 4; mu++)
    for (int nu = mu + 1; nu < 4; nu++, plane++) {
      HC S[4][4];
      for (int r = 0; r < 4; r++)
        for (int q = 0; q < 4; q++) {
          HC acc{0, 0};
          for (int k = 0; k < 4; k++) {
            HC a = hmul(G[mu][r][k], G[nu][k][q]);
            HC b = hmul(G[nu][r][k], G[mu][k][q]);
            acc.re += a.re - b.re;
            acc.im += a.im - b.im;
          }
          S[r][q] = {-0.5 * acc.im, 0.5 * acc.re};  // (i/2) * commutator
        }
      for (int b = 0; b < 2; b++)
        for (int s = 0; s < 2; s++)
          for (int t = 0; t < 2; t++) {
            host[plane][b][s][t][0] = S[2 * b + s][2 * b + t].re;
            host[plane][b][s][t][1] = S[2 * b + s][2 * b + t].im;
          }
      for (int s = 0; s < 2; s++)
        for (int t = 0; t < 2; t++)
          if (std::fabs(S[s][2 + t].re) + std::fabs(S[s][2 + t].im) > 1e-14)
            raise(MG_ERR_ARG, "sigma not block diagonal");
    }
  MG_CUDA(cudaMemcpyToSymbol(c_sigma, host, sizeof(host)));
}
}  // namespace

// --------------------------------------------------------------------------- packing
// nrhs ABI vectors (blockIdx.y) to packed half vectors `stride` elements of T
// apart, the sites of parity blockIdx.z (even_only launches have parity 0
// alone).  A CTA's sites are read as spans of 192 bytes into shared memory
// (16 bytes at a stride of 192 from each thread: 972 us for the even sites of
// twelve vectors of 32^3x64, 873 us so).
constexpr int kPack = 128;   // sites per CTA; rows padded to 13 double2 against bank conflicts
template <typename T>
__global__ void __launch_bounds__(kPack) k_pack_spinor(Geom g, const double2* __restrict__ abi, T* even, T* odd,
                                                       size_t stride) {
  __shared__ double2 sm[kPack * 13];
  __shared__ int slex[kPack];
  const int par = blockIdx.z, cb0 = blockIdx.x * kPack, cb = cb0 + threadIdx.x;
  if (cb < g.Vh) {   // the pair (2 cb, 2 cb + 1) of lexicographic sites has one of each parity
    int r = cb / (g.L[0] / 2), odd_row = r % g.L[1];
    r /= g.L[1];
    odd_row += r % g.L[2] + r / g.L[2];
    slex[threadIdx.x] = 2 * cb + ((odd_row + par) & 1);
  }
  __syncthreads();
  abi += (size_t)blockIdx.y * 24 * g.Vh;
  const int n = 12 * min(kPack, g.Vh - cb0);
#pragma unroll 6
  for (int t = threadIdx.x; t < n; t += kPack) {
    const int i = t / 12, k = t - 12 * i;
    sm[i * 13 + k] = abi[(size_t)slex[i] * 12 + k];
  }
  __syncthreads();
  if (cb >= g.Vh) return;
  cx<T> s[12];
#pragma unroll
  for (int k = 0; k < 12; k++) {
    const double2 v = sm[threadIdx.x * 13 + k];
    s[k] = mkc<T>((T)v.x, (T)v.y);
  }
  SpinorIO<T>::store((par ? odd : even) + blockIdx.y * stride, g.Vh, cb, s);
}

// Packed half vectors to ABI vectors; zero_odd: the odd sites become zero and
// `odd` is not read.  A site's 192 bytes are gathered in shared memory and
// written as one contiguous span per CTA: stored straight from the threads (16
// bytes at a stride of 192) the writes reached 2.2 of 6.7 TB/s.
constexpr int kUnpack = 128;   // sites per CTA; rows padded to 13 double2 against bank conflicts
template <typename T>
__global__ void __launch_bounds__(kUnpack) k_unpack_spinor(Geom g, const T* __restrict__ even,
                                                           const T* __restrict__ odd, double2* __restrict__ abi,
                                                           size_t stride, int zero_odd) {
  __shared__ double2 sm[kUnpack * 13];
  const int lex0 = blockIdx.x * kUnpack, lex = lex0 + threadIdx.x;
  if (lex < 2 * g.Vh) {
    int c[4];
    int r = lex;
    c[0] = r % g.L[0]; r /= g.L[0];
    c[1] = r % g.L[1]; r /= g.L[1];
    c[2] = r % g.L[2]; c[3] = r / g.L[2];
    const int par = (c[0] + c[1] + c[2] + c[3]) & 1;
    cx<T> s[12];
    if (par && zero_odd) {
#pragma unroll
      for (int k = 0; k < 12; k++) s[k] = mkc<T>(0, 0);
    } else {
      SpinorIO<T>::load((par ? odd : even) + blockIdx.y * stride, g.Vh, lex >> 1, s);
    }
#pragma unroll
    for (int k = 0; k < 12; k++) sm[threadIdx.x * 13 + k] = make_double2((double)s[k].re, (double)s[k].im);
  }
  __syncthreads();
  const int n = 12 * min(kUnpack, 2 * g.Vh - lex0);
  double2* dst = abi + (size_t)blockIdx.y * 24 * g.Vh + (size_t)lex0 * 12;
  for (int t = threadIdx.x; t < n; t += kUnpack) dst[t] = sm[(t / 12) * 13 + t % 12];
}

// vectors of one launch: the limit of gridDim.y
constexpr int kMaxVectors = 65535;

void pack_spinors(const Geom& g, int nrhs, const double* abi, void* even, void* odd, size_t stride, bool even_only,
                  bool fp32, cudaStream_t s) {
  auto run = [&](auto* e, auto* o) {
    for (int r0 = 0; r0 < nrhs; r0 += kMaxVectors) {
      const dim3 grid((g.Vh + kPack - 1) / kPack, std::min(nrhs - r0, kMaxVectors), even_only ? 1 : 2);
      k_pack_spinor<<<grid, kPack, 0, s>>>(g, (const double2*)abi + (size_t)r0 * 24 * g.Vh, e + r0 * stride, o + r0 * stride,
                                           stride);
      MG_LAUNCH();
    }
  };
  if (fp32)
    run((float*)even, (float*)odd);
  else
    run((double*)even, (double*)odd);
}

void unpack_spinors(const Geom& g, int nrhs, const void* even, const void* odd, size_t stride, bool zero_odd, bool fp32,
                    double* abi, cudaStream_t s) {
  auto run = [&](auto* e, auto* o) {
    for (int r0 = 0; r0 < nrhs; r0 += kMaxVectors) {
      const dim3 grid((2 * g.Vh + kUnpack - 1) / kUnpack, std::min(nrhs - r0, kMaxVectors));
      k_unpack_spinor<<<grid, kUnpack, 0, s>>>(g, e + r0 * stride, o + r0 * stride, (double2*)abi + (size_t)r0 * 24 * g.Vh,
                                               stride, zero_odd);
      MG_LAUNCH();
    }
  };
  if (fp32)
    run((const float*)even, (const float*)odd);
  else
    run((const double*)even, (const double*)odd);
}

void pack_spinor(const Geom& g, const double* abi, void* even, void* odd, bool fp32, cudaStream_t s) {
  pack_spinors(g, 1, abi, even, odd, 0, false, fp32, s);
}

void unpack_spinor(const Geom& g, const void* even, const void* odd, bool fp32, double* abi, cudaStream_t s) {
  unpack_spinors(g, 1, even, odd, 0, false, fp32, abi, s);
}

__global__ void k_pack_gauge(Geom g, const double2* __restrict__ abi, double2* g64, float2* g32) {
  const int lex = blockIdx.x * blockDim.x + threadIdx.x;
  if (lex >= 2 * g.Vh) return;
  int c[4];
  int r = lex;
  c[0] = r % g.L[0]; r /= g.L[0];
  c[1] = r % g.L[1]; r /= g.L[1];
  c[2] = r % g.L[2]; c[3] = r / g.L[2];
  const int par = (c[0] + c[1] + c[2] + c[3]) & 1;
  const int cb = lex >> 1;
  for (int mu = 0; mu < 4; mu++)
    for (int e = 0; e < 9; e++) {
      double2 v = abi[((size_t)lex * 4 + mu) * 9 + e];
      size_t o = ((size_t)(par * 4 + mu) * 9 + e) * g.Vh + cb;
      g64[o] = v;
      g32[o] = make_float2((float)v.x, (float)v.y);
    }
}

void pack_gauge(const Geom& g, const double* abi, double* g64, float* g32, cudaStream_t s) {
  const int n = 2 * g.Vh, bs = 128;
  k_pack_gauge<<<(n + bs - 1) / bs, bs, 0, s>>>(g, (const double2*)abi, (double2*)g64, (float2*)g32);
  MG_LAUNCH();
}

// --------------------------------------------------------------------------- clover construction
namespace {
typedef cx<double> cd;

__device__ void link_at(const Geom& g, const double* gauge, const int y[4], int mu, cd u[9]) {
  const int par = (y[0] + y[1] + y[2] + y[3]) & 1;
  load_link<double>(gauge, g.Vh, par, mu, cb_index(g, y), u);
}
__device__ void step(const Geom& g, const int x[4], int mu, int d, int y[4]) {
  for (int k = 0; k < 4; k++) y[k] = x[k];
  y[mu] = (x[mu] + d + g.L[mu]) % g.L[mu];
}
// c = a b, a b^dag, a^dag b^dag
__device__ void mm(const cd a[9], const cd b[9], cd c[9]) {
  for (int i = 0; i < 3; i++)
    for (int j = 0; j < 3; j++) {
      cd s = mkc(0.0, 0.0);
      for (int k = 0; k < 3; k++) s = cfma(a[i * 3 + k], b[k * 3 + j], s);
      c[i * 3 + j] = s;
    }
}
__device__ void mmd(const cd a[9], const cd b[9], cd c[9]) {
  for (int i = 0; i < 3; i++)
    for (int j = 0; j < 3; j++) {
      cd s = mkc(0.0, 0.0);
      for (int k = 0; k < 3; k++) s = cfma(a[i * 3 + k], conj(b[j * 3 + k]), s);
      c[i * 3 + j] = s;
    }
}

__device__ void mdmd(const cd a[9], const cd b[9], cd c[9]) {
  for (int i = 0; i < 3; i++)
    for (int j = 0; j < 3; j++) {
      cd s = mkc(0.0, 0.0);
      for (int k = 0; k < 3; k++) s = cfma(b[j * 3 + k], a[k * 3 + i], s);   // (b a)_{j i}
      c[i * 3 + j] = conj(s);
    }
}

// G with G - G^dag = Q_{mu nu}(x) - Q_{mu nu}(x)^dag, Q the sum of the four
// counter-clockwise plaquette leaves at x.  The leaves that run through
// U_nu(x - nu) enter as minus their daggers, so that two leaves at a time share
// their first or last link: ten products instead of twelve.
__device__ void clover_leaves(const Geom& g, const double* gauge, const int x[4], int mu, int nu, cd q[9]) {
  int xm[4], xn[4], y[4];
  cd a[9], b[9], t[9], u[9];
  // U_mu(x) [U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag - U_nu(x-nu+mu)^dag U_mu(x-nu)^dag U_nu(x-nu)]
  step(g, x, mu, +1, xm); link_at(g, gauge, xm, nu, a);
  step(g, x, nu, +1, y); link_at(g, gauge, y, mu, b);
  mmd(a, b, t);
  link_at(g, gauge, x, nu, a);
  mmd(t, a, u);
  step(g, xm, nu, -1, y); link_at(g, gauge, y, nu, a);
  step(g, x, nu, -1, xn); link_at(g, gauge, xn, mu, b);
  mdmd(a, b, t);
  link_at(g, gauge, xn, nu, a);
  mm(t, a, b);
  for (int e = 0; e < 9; e++) u[e] = u[e] - b[e];
  link_at(g, gauge, x, mu, a);
  mm(a, u, q);
  // [U_nu(x) U_mu(x+nu-mu)^dag U_nu(x-mu)^dag - U_nu(x-nu)^dag U_mu(x-mu-nu)^dag U_nu(x-mu-nu)] U_mu(x-mu)
  step(g, x, mu, -1, xm);
  link_at(g, gauge, x, nu, a);
  step(g, xm, nu, +1, y); link_at(g, gauge, y, mu, b);
  mmd(a, b, t);
  link_at(g, gauge, xm, nu, a);
  mmd(t, a, u);
  link_at(g, gauge, xn, nu, a);
  step(g, xm, nu, -1, y); link_at(g, gauge, y, mu, b);
  mdmd(a, b, t);
  link_at(g, gauge, y, nu, a);
  mm(t, a, b);
  for (int e = 0; e < 9; e++) u[e] = u[e] - b[e];
  link_at(g, gauge, xm, mu, a);
  mm(u, a, t);
  for (int e = 0; e < 9; e++) q[e] = q[e] + t[e];
}

// Inverse of a 6x6 complex matrix by Gauss-Jordan with partial pivoting, in
// place (the columns of the inverse replace the eliminated ones, the row
// exchanges become column exchanges at the end) and in registers: every index
// is a constant, an exchange is a select.  Returns false if a pivot falls below
// 1e-12 of the largest entry.
__device__ __forceinline__ bool invert6(cd (&m)[36]) {
  double amax = 0;
#pragma unroll
  for (int e = 0; e < 36; e++) amax = fmax(amax, fabs(m[e].re) + fabs(m[e].im));
  bool ok = amax > 0;
  int perm[6];
#pragma unroll
  for (int col = 0; col < 6; col++) {
    int piv = col;
    double best = -1;
#pragma unroll
    for (int r = col; r < 6; r++) {
      const double v = fma(m[r * 6 + col].re, m[r * 6 + col].re, m[r * 6 + col].im * m[r * 6 + col].im);
      if (v > best) { best = v; piv = r; }
    }
    perm[col] = piv;
    if (!(sqrt(best) > 1e-12 * amax)) { ok = false; best = 1.0; }
#pragma unroll
    for (int r = col + 1; r < 6; r++)
      if (piv == r) {
#pragma unroll
        for (int j = 0; j < 6; j++) {
          const cd t = m[col * 6 + j];
          m[col * 6 + j] = m[r * 6 + j];
          m[r * 6 + j] = t;
        }
      }
    const cd p = m[col * 6 + col];
    double den = fma(p.re, p.re, p.im * p.im);
    if (den == 0) den = 1;
    const double di = 1.0 / den;
    const cd pinv = mkc(p.re * di, -p.im * di);
#pragma unroll
    for (int j = 0; j < 6; j++) m[col * 6 + j] = j == col ? pinv : pinv * m[col * 6 + j];
#pragma unroll
    for (int r = 0; r < 6; r++) {
      if (r == col) continue;
      const cd f = m[r * 6 + col], nf = mkc(-f.re, -f.im);
#pragma unroll
      for (int j = 0; j < 6; j++) m[r * 6 + j] = j == col ? nf * m[col * 6 + j] : cfma(nf, m[col * 6 + j], m[r * 6 + j]);
    }
  }
#pragma unroll
  for (int col = 5; col >= 0; col--)
#pragma unroll
    for (int r = col + 1; r < 6; r++)
      if (perm[col] == r) {
#pragma unroll
        for (int i = 0; i < 6; i++) {
          const cd t = m[i * 6 + col];
          m[i * 6 + col] = m[i * 6 + r];
          m[i * 6 + r] = t;
        }
      }
  return ok;
}

__device__ __forceinline__ void pack_herm(const cd (&m)[36], double (&r)[36]) {
#pragma unroll
  for (int i = 0; i < 6; i++) r[i] = m[i * 6 + i].re;
#pragma unroll
  for (int i = 1; i < 6; i++)
#pragma unroll
    for (int j = 0; j < i; j++) {
      const int k = i * (i - 1) / 2 + j;
      r[6 + 2 * k] = m[i * 6 + j].re;
      r[6 + 2 * k + 1] = m[i * 6 + j].im;
    }
}
}  // namespace

// One thread per site, bound by the FP64 pipe: per plane ten 3x3 products, per
// spin entry of sigma one product with F (the zero entries are skipped, the
// condition is the same for all threads), and two inversions in place.  With
// twelve products, two complex products per entry and the inversion of the
// augmented matrix in local memory 131072 sites took 4.11 ms, 2.41 here.
__global__ void __launch_bounds__(64) k_build_clover(Geom g, const double* __restrict__ gauge, CloverCoef cf, double m0,
                                                     double* A64, double* Ainv64, float* A32, float* Ainv32,
                                                     int* flags) {
  const int gid = blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= 2 * g.Vh) return;
  const int par = gid / g.Vh, i = gid % g.Vh;
  int x[4];
  cb_coords(g, i, par, x);
  // lower triangles (i >= j) of the two chiral blocks
  cd L[2][21];
#pragma unroll
  for (int b = 0; b < 2; b++)
#pragma unroll
    for (int e = 0; e < 21; e++) L[b][e] = mkc(0.0, 0.0);
  int plane = 0;
#pragma unroll 1
  for (int mu = 0; mu < 4; mu++)
#pragma unroll 1
    for (int nu = mu + 1; nu < 4; nu++, plane++) {
      cd q[9], F[9];
      clover_leaves(g, gauge, x, mu, nu, q);
#pragma unroll
      for (int a = 0; a < 3; a++)
#pragma unroll
        for (int c = 0; c < 3; c++) F[a * 3 + c] = 0.125 * (q[a * 3 + c] - conj(q[c * 3 + a]));
      const cd tr = mkc((F[0].re + F[4].re + F[8].re) / 3.0, (F[0].im + F[4].im + F[8].im) / 3.0);
      F[0] = F[0] - tr; F[4] = F[4] - tr; F[8] = F[8] - tr;
      // sum over mu != nu of both orders gives 2x the mu < nu term:
      // A += (i c_{mu nu} / 2) sigma_{mu nu} (x) F_{mu nu}, c = csw_t for the planes
      // that contain t, csw_s for the spatial ones (one csw when isotropic)
      const double pre = 0.5 * (nu == 3 ? cf.csw_t : cf.csw_s);
#pragma unroll
      for (int b = 0; b < 2; b++)
#pragma unroll
        for (int si = 0; si < 2; si++)
#pragma unroll
          for (int sj = 0; sj <= si; sj++) {
            const cd sg = mkc(-pre * c_sigma[plane][b][si][sj][1], pre * c_sigma[plane][b][si][sj][0]);   // i pre sigma
            if (sg.re == 0.0 && sg.im == 0.0) continue;
#pragma unroll
            for (int ci = 0; ci < 3; ci++)
#pragma unroll
              for (int cj = 0; cj < 3; cj++) {
                const int ii = 3 * si + ci, jj = 3 * sj + cj;
                if (jj > ii) continue;
                cd& e = L[b][ii * (ii + 1) / 2 + jj];
                e = cfma(sg, F[ci * 3 + cj], e);
              }
          }
    }
  bool ok = true;
#pragma unroll
  for (int b = 0; b < 2; b++) {
    cd M[36];
#pragma unroll
    for (int ii = 0; ii < 6; ii++)
#pragma unroll
      for (int jj = 0; jj <= ii; jj++) {
        cd v = L[b][ii * (ii + 1) / 2 + jj];
        if (ii == jj) v = mkc(v.re + (g.w[0] + g.w[1] + g.w[2] + g.w[3]) + m0, 0.0);   // 4 + m0 when isotropic
        M[ii * 6 + jj] = v;
        M[jj * 6 + ii] = conj(v);
      }
    double r[36];
    float rf[36];
    pack_herm(M, r);
    CloverIO<double>::store_block(A64 + (size_t)par * 72 * g.Vh, g.Vh, i, b, r);
#pragma unroll
    for (int e = 0; e < 36; e++) rf[e] = (float)r[e];
    CloverIO<float>::store_block(A32 + (size_t)par * 72 * g.Vh, g.Vh, i, b, rf);
    ok &= invert6(M);
    // symmetrise: store the Hermitian part of the inverse
#pragma unroll
    for (int ii = 0; ii < 6; ii++)
#pragma unroll
      for (int jj = 0; jj <= ii; jj++) {
        const cd a = M[ii * 6 + jj], c = conj(M[jj * 6 + ii]);
        M[ii * 6 + jj] = mkc(0.5 * (a.re + c.re), 0.5 * (a.im + c.im));
      }
    pack_herm(M, r);
    CloverIO<double>::store_block(Ainv64 + (size_t)par * 72 * g.Vh, g.Vh, i, b, r);
#pragma unroll
    for (int e = 0; e < 36; e++) rf[e] = (float)r[e];
    CloverIO<float>::store_block(Ainv32 + (size_t)par * 72 * g.Vh, g.Vh, i, b, rf);
  }
  if (!ok) atomicExch(&flags[FLAG_SINGULAR], 1);
}

void build_clover(const Geom& g, const double* g64, CloverCoef cf, double m0, double* A64, double* Ainv64,
                  float* A32, float* Ainv32, int* flags, cudaStream_t s) {
  upload_sigma();
  const int n = 2 * g.Vh, bs = 64;
  k_build_clover<<<(n + bs - 1) / bs, bs, 0, s>>>(g, g64, cf, m0, A64, Ainv64, A32, Ainv32, flags);
  MG_LAUNCH();
}

// --------------------------------------------------------------------------- clover apply
template <typename T>
__global__ void k_clover_apply(Geom g, T* out, const T* __restrict__ in, const T* __restrict__ clov) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.Vh) return;
  cx<T> x[12], y[12];
  SpinorIO<T>::load(in, g.Vh, i, x);
  clover_mul<T>(clov, g.Vh, i, x, y);
  SpinorIO<T>::store(out, g.Vh, i, y);
}

template <typename T>
void clover_apply(const Geom& g, T* out, const T* in, const T* clov, cudaStream_t s) {
  const int bs = site_block(g.Vh);
  k_clover_apply<T><<<(g.Vh + bs - 1) / bs, bs, 0, s>>>(g, out, in, clov);
  MG_LAUNCH();
}
template void clover_apply<float>(const Geom&, float*, const float*, const float*, cudaStream_t);
template void clover_apply<double>(const Geom&, double*, const double*, const double*, cudaStream_t);

// --------------------------------------------------------------------------- dslash
// One output site: out = epilogue(-1/2 H in) (see Epilogue).
template <typename T, int EPI>
__device__ __forceinline__ void dslash_site(const Geom& g, int par, int i, T* out, const T* __restrict__ in,
                                            const T* __restrict__ gauge, const T* __restrict__ clov,
                                            const T* __restrict__ x, T a, int dirmask) {
  int c[4];
  cb_coords(g, i, par, c);
  cx<T> acc[12];
#pragma unroll
  for (int k = 0; k < 12; k++) acc[k] = mkc<T>(0, 0);
  hop_sum<T>(g, in, gauge, par, i, c, dirmask, acc);
  const T half = (T)-0.5;
  cx<T> res[12];
  if (EPI == EPI_H) {
#pragma unroll
    for (int k = 0; k < 12; k++) res[k] = half * acc[k];
  } else if (EPI == EPI_CH) {
#pragma unroll
    for (int k = 0; k < 12; k++) acc[k] = half * acc[k];
    clover_mul<T>(clov, g.Vh, i, acc, res);
  } else if (EPI == EPI_XPAY) {
    cx<T> xv[12];
    SpinorIO<T>::load(x, g.Vh, i, xv);
    const T f = half * a;
#pragma unroll
    for (int k = 0; k < 12; k++) res[k] = xv[k] + f * acc[k];
  } else if (EPI == EPI_CX_PAY) {
    cx<T> xv[12];
    SpinorIO<T>::load(x, g.Vh, i, xv);
    clover_mul<T>(clov, g.Vh, i, xv, res);
    const T f = half * a;
#pragma unroll
    for (int k = 0; k < 12; k++) res[k] = res[k] + f * acc[k];
  } else {  // EPI_C_XPAY
    cx<T> xv[12];
    SpinorIO<T>::load(x, g.Vh, i, xv);
    const T f = half * a;
#pragma unroll
    for (int k = 0; k < 12; k++) xv[k] = xv[k] + f * acc[k];
    clover_mul<T>(clov, g.Vh, i, xv, res);
  }
  SpinorIO<T>::store(out, g.Vh, i, res);
}

// Operands of the output parities par0 + blockIdx.y, indexed by parity (`in`
// is the half of the other parity).
template <typename T>
struct HalfArgs {
  T* out[2];
  const T* in[2];
  const T* clov[2];
  const T* x[2];
};
template <typename T, int EPI>
__global__ void __launch_bounds__(128) k_dslash(Geom g, int par0, HalfArgs<T> h, const T* __restrict__ gauge, T a,
                                                int dirmask) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.Vh) return;
  const int par = par0 + blockIdx.y;
  dslash_site<T, EPI>(g, par, i, par ? h.out[1] : h.out[0], par ? h.in[1] : h.in[0], gauge,
                      par ? h.clov[1] : h.clov[0], par ? h.x[1] : h.x[0], a, dirmask);
}

// The same for lattices that do not fill the GPU: four lanes per site
// (wilson_dev.cuh), 32 sites and 128 threads or 8 and 32 per CTA.
template <typename T, int EPI>
__global__ void __launch_bounds__(128) k_dslash_lanes(Geom g, int par0, HalfArgs<T> h, const T* __restrict__ gauge,
                                                       T a) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int k = t & 1, b = (t >> 1) & 1, s = 2 * b + k;
  const bool live = (t >> 2) < g.Vh;
  const int i = live ? t >> 2 : g.Vh - 1;   // every lane takes part in the shuffles
  const int par = par0 + blockIdx.y;
  const T* clov = par ? h.clov[1] : h.clov[0];
  const T* x = par ? h.x[1] : h.x[0];
  cx<T> acc[3], xv[3], res[3];
  if (EPI != EPI_H && EPI != EPI_CH) {
#pragma unroll
    for (int r = 0; r < 3; r++) xv[r] = SpinorIO<T>::get(x, g.Vh, i, 3 * s + r);
  }
  lane_hop_sum<T>(g, par ? h.in[1] : h.in[0], gauge, par, i, k, b, acc);
  const T half = (T)-0.5, f = half * a;
  if (EPI == EPI_H || EPI == EPI_CH) {
#pragma unroll
    for (int r = 0; r < 3; r++) res[r] = half * acc[r];
    if (EPI == EPI_CH) {
#pragma unroll
      for (int r = 0; r < 3; r++) acc[r] = res[r];
      lane_clover<T>(clov, g.Vh, i, k, b, acc, res);
    }
  } else if (EPI == EPI_CX_PAY) {
    lane_clover<T>(clov, g.Vh, i, k, b, xv, res);
#pragma unroll
    for (int r = 0; r < 3; r++) res[r] = res[r] + f * acc[r];
  } else {
#pragma unroll
    for (int r = 0; r < 3; r++) xv[r] = xv[r] + f * acc[r];
    if (EPI == EPI_C_XPAY) {
      lane_clover<T>(clov, g.Vh, i, k, b, xv, res);
    } else {
#pragma unroll
      for (int r = 0; r < 3; r++) res[r] = xv[r];
    }
  }
  if (live) {
    T* out = par ? h.out[1] : h.out[0];
#pragma unroll
    for (int r = 0; r < 3; r++) SpinorIO<T>::put(out, g.Vh, i, 3 * s + r, res[r]);
  }
}

// The epilogues of the multi-RHS kernels for the nr <= NR right-hand sides
// r0 .. r0 + nr - 1 of site i (acc: the hop sums without the -1/2).
template <typename T, int EPI, int NR>
__device__ __forceinline__ void mrhs_epilogue(const Geom& g, int i, cx<T> (&acc)[NR][12], int nr, int r0,
                                              size_t stride, T* out, const T* __restrict__ clov,
                                              const T* __restrict__ x, T a) {
  const T half = (T)-0.5;
#pragma unroll
  for (int r = 0; r < NR; r++) {
    if (r >= nr) break;
    const size_t o = (size_t)(r0 + r) * stride;
    cx<T> res[12];
    if (EPI == EPI_H) {
#pragma unroll
      for (int k = 0; k < 12; k++) res[k] = half * acc[r][k];
    } else if (EPI == EPI_CH) {
#pragma unroll
      for (int k = 0; k < 12; k++) acc[r][k] = half * acc[r][k];
      clover_mul<T>(clov, g.Vh, i, acc[r], res);
    } else if (EPI == EPI_XPAY) {
      cx<T> xv[12];
      SpinorIO<T>::load(x + o, g.Vh, i, xv);
      const T f = half * a;
#pragma unroll
      for (int k = 0; k < 12; k++) res[k] = xv[k] + f * acc[r][k];
    } else if (EPI == EPI_CX_PAY) {
      cx<T> xv[12];
      SpinorIO<T>::load(x + o, g.Vh, i, xv);
      clover_mul<T>(clov, g.Vh, i, xv, res);
      const T f = half * a;
#pragma unroll
      for (int k = 0; k < 12; k++) res[k] = res[k] + f * acc[r][k];
    } else {  // EPI_C_XPAY
      cx<T> xv[12];
      SpinorIO<T>::load(x + o, g.Vh, i, xv);
      const T f = half * a;
#pragma unroll
      for (int k = 0; k < 12; k++) xv[k] = xv[k] + f * acc[r][k];
      clover_mul<T>(clov, g.Vh, i, xv, res);
    }
    SpinorIO<T>::store(out + o, g.Vh, i, res);
  }
}

// Multi-RHS form: nrhs vectors at a fixed stride (in elements of T).  A
// thread owns one site and NR right-hand sides (the block index selects the
// site block and the group of NR, group fastest): every link is loaded once
// into registers and applied to the NR
// neighbour spinors, so link bytes are paid once per site and NR rhs while
// the spinor loads stay coalesced over consecutive sites.
template <typename T, int EPI, int NR, int BS, int MINB>
__global__ void __launch_bounds__(BS, MINB) k_dslash_mrhs(Geom g, int par, int nrhs, size_t stride, T* out,
                                                    const T* __restrict__ in, const T* __restrict__ gauge,
                                                    const T* __restrict__ clov, const T* __restrict__ x, T a,
                                                    int dirmask) {
  // 1-D grid, rhs group fastest: CTAs that run together share the sites
  // (and so the link and clover lines in L2) of consecutive rhs groups
  const int ngroups = (nrhs + NR - 1) / NR;
  const int i = (int)(blockIdx.x / ngroups) * BS + threadIdx.x;
  if (i >= g.Vh) return;
  const int r0 = (int)(blockIdx.x % ngroups) * NR;
  const int nr = nrhs - r0 < NR ? nrhs - r0 : NR;
  int c[4];
  cb_coords(g, i, par, c);
  cx<T> acc[NR][12];
#pragma unroll
  for (int r = 0; r < NR; r++)
#pragma unroll
    for (int k = 0; k < 12; k++) acc[r][k] = mkc<T>(0, 0);
  hop_sum_nr<T, NR>(g, in + (size_t)r0 * stride, stride, nr, gauge, par, i, c, dirmask, acc);
  mrhs_epilogue<T, EPI, NR>(g, i, acc, nr, r0, stride, out, clov, x, a);
}

// Threads per CTA of the one-site-per-thread kernels for `ctas128` CTAs of 128
// sites: the largest of 128, 64, 32 that gives every SM about six CTAs or more
// (below that the last wave leaves SMs idle: 65536 sites in CTAs of 128 are 3.4
// per SM, so some SMs take 4 and some 3; 4096 sites used 32 of 152 SMs, and in
// FP64 a busy SM then runs at its FP64 rate while the others idle: 45 us for
// 960 sites).
int site_block(long long sites) { return sites >= 128 * 152 * 6 ? 128 : sites >= 64 * 152 * 6 ? 64 : 32; }

// Four lanes per site, by the sites of a launch (both parities where it has both).
// FP64: by the length of the busiest scheduler's chain (608 schedulers; a warp of 32
// sites is about 1320 FP64 instructions of 64 cycles each, one of 8 sites and four
// lanes each about 380).  Lanes / a thread per site: 15.8 / 43.5 us at 1920 sites,
// 35 / 44 at 12288, 50 / 46 at 18432, 111 / 117 at 41472, 256 / 260 at 98304, 329 / 303
// at 131072; one parity 21.8 / 35.7 at 9216, 52 / 57 at 20736, 72 / 66 at 32768, 111 /
// 101 at 49152.  FP32, up to kLanesF32 sites, where latency and not bandwidth sets the
// time: 5.2 / 7.0 us at 8192 sites, 6.3 / 7.7 at 18432, 7.9 / 7.8 at 27648, 11.6 / 8.9
// at 41472; one parity 4.3 / 5.8 at 4096, 6.1 / 6.9 at 20736, 7.7 / 7.3 at 32768.
constexpr int kLanesF32 = 24576;
template <typename T>
bool lanes_per_site(int sites) {
  if (sizeof(T) == 4) return sites <= kLanesF32;
  const int warps = (sites + 31) / 32;
  return ((4 * warps + 607) / 608) * 380 < ((warps + 607) / 608) * 1320;
}

bool dslash_lanes_f32(int Vh) { return lanes_per_site<float>(Vh); }

template <typename T>
void dslash_halves(const Geom& g, Epilogue epi, int par0, int npar, const HalfArgs<T>& h, const T* gauge, double a,
                   int dirmask, cudaStream_t s) {
  if (dirmask == 0xff && lanes_per_site<T>(npar * g.Vh)) {
    const int bl = site_block((long long)g.Vh * 4);
    const dim3 nl((4 * g.Vh + bl - 1) / bl, npar);
    switch (epi) {
      case EPI_H: k_dslash_lanes<T, EPI_H><<<nl, bl, 0, s>>>(g, par0, h, gauge, (T)a); break;
      case EPI_CH: k_dslash_lanes<T, EPI_CH><<<nl, bl, 0, s>>>(g, par0, h, gauge, (T)a); break;
      case EPI_XPAY: k_dslash_lanes<T, EPI_XPAY><<<nl, bl, 0, s>>>(g, par0, h, gauge, (T)a); break;
      case EPI_CX_PAY: k_dslash_lanes<T, EPI_CX_PAY><<<nl, bl, 0, s>>>(g, par0, h, gauge, (T)a); break;
      case EPI_C_XPAY: k_dslash_lanes<T, EPI_C_XPAY><<<nl, bl, 0, s>>>(g, par0, h, gauge, (T)a); break;
    }
    MG_LAUNCH();
    return;
  }
  const int bs = site_block((long long)g.Vh * npar);
  const dim3 nb((g.Vh + bs - 1) / bs, npar);
  switch (epi) {
    case EPI_H: k_dslash<T, EPI_H><<<nb, bs, 0, s>>>(g, par0, h, gauge, (T)a, dirmask); break;
    case EPI_CH: k_dslash<T, EPI_CH><<<nb, bs, 0, s>>>(g, par0, h, gauge, (T)a, dirmask); break;
    case EPI_XPAY: k_dslash<T, EPI_XPAY><<<nb, bs, 0, s>>>(g, par0, h, gauge, (T)a, dirmask); break;
    case EPI_CX_PAY: k_dslash<T, EPI_CX_PAY><<<nb, bs, 0, s>>>(g, par0, h, gauge, (T)a, dirmask); break;
    case EPI_C_XPAY: k_dslash<T, EPI_C_XPAY><<<nb, bs, 0, s>>>(g, par0, h, gauge, (T)a, dirmask); break;
  }
  MG_LAUNCH();
}

template <typename T>
void dslash(const Geom& g, Epilogue epi, int parity, T* out, const T* in, const T* gauge, const T* clov, const T* x,
            double a, int dirmask, cudaStream_t s) {
  HalfArgs<T> h{{out, out}, {in, in}, {clov, clov}, {x, x}};
  dslash_halves<T>(g, epi, parity, 1, h, gauge, a, dirmask, s);
}

template <typename T>
void dslash_full(const Geom& g, Epilogue epi, T* oe, T* oo, const T* ie, const T* io, const T* gauge, const T* ce,
                 const T* co, const T* xe, const T* xo, double a, cudaStream_t s) {
  HalfArgs<T> h{{oe, oo}, {io, ie}, {ce, co}, {xe, xo}};
  dslash_halves<T>(g, epi, 0, 2, h, gauge, a, 0xff, s);
}
template void dslash_full<float>(const Geom&, Epilogue, float*, float*, const float*, const float*, const float*,
                                 const float*, const float*, const float*, const float*, double, cudaStream_t);
template void dslash_full<double>(const Geom&, Epilogue, double*, double*, const double*, const double*, const double*,
                                  const double*, const double*, const double*, const double*, double, cudaStream_t);
template void dslash<float>(const Geom&, Epilogue, int, float*, const float*, const float*, const float*,
                            const float*, double, int, cudaStream_t);
template void dslash<double>(const Geom&, Epilogue, int, double*, const double*, const double*, const double*,
                             const double*, double, int, cudaStream_t);

// Second mapping: one (site, rhs) per thread, the CTA is 32 consecutive sites
// (threadIdx.x) x NY right-hand sides (threadIdx.y).  Each warp reads 32
// consecutive sites of one rhs (coalesced spinors) with the register
// footprint of the single-RHS kernel; the NY warps of a CTA read the same
// link and clover lines, which the first one brings into L1.
template <typename T, int EPI, int NY>
__global__ void __launch_bounds__(32 * NY) k_dslash_mrhs_y(Geom g, int par, int nrhs, size_t stride, T* out,
                                                            const T* __restrict__ in, const T* __restrict__ gauge,
                                                            const T* __restrict__ clov, const T* __restrict__ x, T a,
                                                            int dirmask) {
  const int ngroups = (nrhs + NY - 1) / NY;   // rhs group fastest in the 1-D grid
  const int i = (int)(blockIdx.x / ngroups) * 32 + threadIdx.x;
  const int r = (int)(blockIdx.x % ngroups) * NY + threadIdx.y;
  if (i >= g.Vh || r >= nrhs) return;
  const size_t o = (size_t)r * stride;
  dslash_site<T, EPI>(g, par, i, out + o, in + o, gauge, clov, x ? x + o : nullptr, a, dirmask);
}

template <typename T, int NY>
void dslash_mrhs_y(const Geom& g, Epilogue epi, int parity, int nrhs, size_t stride, T* out, const T* in,
                   const T* gauge, const T* clov, const T* x, double a, int dirmask, cudaStream_t s) {
  const dim3 grid((unsigned)(((g.Vh + 31) / 32) * ((nrhs + NY - 1) / NY))), block(32, NY);
  switch (epi) {
    case EPI_H: k_dslash_mrhs_y<T, EPI_H, NY><<<grid, block, 0, s>>>(g, parity, nrhs, stride, out, in, gauge, clov, x, (T)a, dirmask); break;
    case EPI_CH: k_dslash_mrhs_y<T, EPI_CH, NY><<<grid, block, 0, s>>>(g, parity, nrhs, stride, out, in, gauge, clov, x, (T)a, dirmask); break;
    case EPI_XPAY: k_dslash_mrhs_y<T, EPI_XPAY, NY><<<grid, block, 0, s>>>(g, parity, nrhs, stride, out, in, gauge, clov, x, (T)a, dirmask); break;
    case EPI_CX_PAY: k_dslash_mrhs_y<T, EPI_CX_PAY, NY><<<grid, block, 0, s>>>(g, parity, nrhs, stride, out, in, gauge, clov, x, (T)a, dirmask); break;
    case EPI_C_XPAY: k_dslash_mrhs_y<T, EPI_C_XPAY, NY><<<grid, block, 0, s>>>(g, parity, nrhs, stride, out, in, gauge, clov, x, (T)a, dirmask); break;
  }
  MG_LAUNCH();
}

// Third mapping (FP32): the CTA stages the links of its S consecutive output
// sites -- both hops of every dimension, 8 x 9 complex per site -- and, when
// the epilogue multiplies by a clover term, that term (18 float4 per site) in
// shared memory once, and then runs every right-hand side over them: thread
// (s, q) owns site s and the right-hand sides q, q + NQ, ...  Link and clover
// bytes leave L2 once per site for all nrhs (not once per rhs group), the
// neighbour spinors are read per rhs exactly as by the single-RHS kernel, and
// each thread keeps the single-RHS register footprint.
constexpr bool epi_has_clover(int epi) { return epi == EPI_CH || epi == EPI_CX_PAY || epi == EPI_C_XPAY; }

template <int S>
__device__ __forceinline__ void clover_mul_smem(const float4* sc, int s, const cx<float> x[12], cx<float> y[12]) {
#pragma unroll
  for (int b = 0; b < 2; b++) {
    float r[36];
#pragma unroll
    for (int k = 0; k < 9; k++) {
      const float4 v = sc[(9 * b + k) * S + s];
      r[4 * k] = v.x;
      r[4 * k + 1] = v.y;
      r[4 * k + 2] = v.z;
      r[4 * k + 3] = v.w;
    }
    herm6_apply<float>(r, x + 6 * b, y + 6 * b);
  }
}

// hop D (D = 2 mu + 1 for the backward hop) of one rhs with its link from shared memory
template <int D, int S>
__device__ __forceinline__ void smem_hop(const Geom& g, const float* __restrict__ in, const float2* sl, int s, int j,
                                         float sgw, cx<float> acc[12]) {
  cx<float> psi[12];
  SpinorIO<float>::load(in, g.Vh, j, psi);
  cx<float> u[9];
#pragma unroll
  for (int e = 0; e < 9; e++) {
    const float2 v = sl[(D * 9 + e) * S + s];
    u[e] = mkc(v.x, v.y);
  }
  hop_apply<float, D / 2, (D & 1) == 0>(psi, u, sgw, acc);
}

template <int D>
__device__ __forceinline__ int dir_bit() { return (D & 1) ? 16 << (D / 2) : 1 << (D / 2); }

// Site block of the CTA launched as `b`.  Natural order (tt == 0): block b.
// Tiled order (tt > 0, which needs S to divide the xh Ly sites of a (z, t)
// plane -- nyb blocks per plane -- and tt to divide Lt): the lattice is cut
// into slabs of tt time slices, taken one after the other; inside a slab the
// blocks of a plane come first, then the next time slice, then the next z.
// A neighbour in t is then nyb launches away and one in z nyb * tt launches
// away, instead of a whole time slice (Vh / Lt sites) for t: with all
// right-hand sides of a site in flight at once, the spinors of a time slice
// no longer fit in L2 between their uses, those of a slab's window do.
__device__ __forceinline__ int mrhs_block(const Geom& g, int b, int nyb, int tt) {
  if (tt <= 0) return b;
  const int yb = b % nyb;
  int r = b / nyb;
  const int tin = r % tt;
  r /= tt;
  const int z = r % g.L[2];
  const int t = (r / g.L[2]) * tt + tin;
  return yb + nyb * (z + g.L[2] * t);
}

template <int EPI, int S, int NQ, int MINB>
__global__ void __launch_bounds__(S * NQ, MINB) k_dslash_mrhs_smem(Geom g, int par, int nrhs, size_t stride,
                                                                    float* out, const float* __restrict__ in,
                                                                    const float* __restrict__ gauge,
                                                                    const float* __restrict__ clov,
                                                                    const float* __restrict__ x, float a, int dirmask,
                                                                    int nyb, int tt) {
  extern __shared__ float4 dsm[];
  float2* sl = reinterpret_cast<float2*>(dsm);   // [8 hops][9][S]
  float4* sc = dsm + 36 * S;                      // [18][S], after the 72 S float2 of links
  __shared__ int snb[8][S];                       // neighbour index of every hop of the CTA's sites
  __shared__ float ssg[8][S];                     // boundary sign x hopping weight of every hop
  const int s = (int)threadIdx.x % S, q = (int)threadIdx.x / S;
  const int i = mrhs_block(g, (int)blockIdx.x, nyb, tt) * S + s;
  const bool valid = i < g.Vh;
  if (valid) {
    int c[4];
    cb_coords(g, i, par, c);
    int nb[8];
    float sg[8];
    int sgn;
#define MG_SMEM_NB(D, MU, FWD)                \
  nb[D] = neighbour<MU, FWD>(g, c, sgn);        \
  sg[D] = (float)sgn * (float)g.w[MU];
    MG_SMEM_NB(0, 0, true) MG_SMEM_NB(1, 0, false) MG_SMEM_NB(2, 1, true) MG_SMEM_NB(3, 1, false)
    MG_SMEM_NB(4, 2, true) MG_SMEM_NB(5, 2, false) MG_SMEM_NB(6, 3, true) MG_SMEM_NB(7, 3, false)
#undef MG_SMEM_NB
    if (q == 0) {
#pragma unroll
      for (int d = 0; d < 8; d++) {
        snb[d][s] = nb[d];
        ssg[d][s] = sg[d];
      }
    }
    // links: U_mu(x) of this parity for the forward hops, U_mu(x - mu) of the
    // other parity for the backward ones
    const float2* gl = reinterpret_cast<const float2*>(gauge);
#pragma unroll
    for (int d = 0; d < 8; d++) {
      const int bit = (d & 1) ? 16 << (d / 2) : 1 << (d / 2);
      if (d % NQ != q || !(dirmask & bit)) continue;
      const int site = (d & 1) ? nb[d] : i;
      const float2* p = gl + (size_t)((((d & 1) ? 1 - par : par) * 4) + d / 2) * 9 * g.Vh;
#pragma unroll
      for (int e = 0; e < 9; e++) sl[(d * 9 + e) * S + s] = p[(size_t)e * g.Vh + site];
    }
    if (epi_has_clover(EPI)) {
      const float4* cp = reinterpret_cast<const float4*>(clov);
      for (int k = q; k < 18; k += NQ) sc[k * S + s] = cp[(size_t)k * g.Vh + i];
    }
  }
  __syncthreads();
  if (!valid) return;
  const float half = -0.5f;
  for (int r = q; r < nrhs; r += NQ) {
    const size_t o = (size_t)r * stride;
    const float* inr = in + o;
    cx<float> acc[12];
#pragma unroll
    for (int k = 0; k < 12; k++) acc[k] = mkc<float>(0, 0);
    if (dirmask & dir_bit<0>()) smem_hop<0, S>(g, inr, sl, s, snb[0][s], ssg[0][s], acc);
    if (dirmask & dir_bit<1>()) smem_hop<1, S>(g, inr, sl, s, snb[1][s], ssg[1][s], acc);
    if (dirmask & dir_bit<2>()) smem_hop<2, S>(g, inr, sl, s, snb[2][s], ssg[2][s], acc);
    if (dirmask & dir_bit<3>()) smem_hop<3, S>(g, inr, sl, s, snb[3][s], ssg[3][s], acc);
    if (dirmask & dir_bit<4>()) smem_hop<4, S>(g, inr, sl, s, snb[4][s], ssg[4][s], acc);
    if (dirmask & dir_bit<5>()) smem_hop<5, S>(g, inr, sl, s, snb[5][s], ssg[5][s], acc);
    if (dirmask & dir_bit<6>()) smem_hop<6, S>(g, inr, sl, s, snb[6][s], ssg[6][s], acc);
    if (dirmask & dir_bit<7>()) smem_hop<7, S>(g, inr, sl, s, snb[7][s], ssg[7][s], acc);
    cx<float> res[12];
    if (EPI == EPI_H) {
#pragma unroll
      for (int k = 0; k < 12; k++) res[k] = half * acc[k];
    } else if (EPI == EPI_CH) {
#pragma unroll
      for (int k = 0; k < 12; k++) acc[k] = half * acc[k];
      clover_mul_smem<S>(sc, s, acc, res);
    } else if (EPI == EPI_XPAY) {
      cx<float> xv[12];
      SpinorIO<float>::load(x + o, g.Vh, i, xv);
      const float f = half * a;
#pragma unroll
      for (int k = 0; k < 12; k++) res[k] = xv[k] + f * acc[k];
    } else if (EPI == EPI_CX_PAY) {
      cx<float> xv[12];
      SpinorIO<float>::load(x + o, g.Vh, i, xv);
      clover_mul_smem<S>(sc, s, xv, res);
      const float f = half * a;
#pragma unroll
      for (int k = 0; k < 12; k++) res[k] = res[k] + f * acc[k];
    } else {  // EPI_C_XPAY
      cx<float> xv[12];
      SpinorIO<float>::load(x + o, g.Vh, i, xv);
      const float f = half * a;
#pragma unroll
      for (int k = 0; k < 12; k++) xv[k] = xv[k] + f * acc[k];
      clover_mul_smem<S>(sc, s, xv, res);
    }
    SpinorIO<float>::store(out + o, g.Vh, i, res);
  }
}

template <int EPI, int S, int NQ, int MINB>
void launch_mrhs_smem(const Geom& g, int parity, int nrhs, size_t stride, float* out, const float* in,
                      const float* gauge, const float* clov, const float* x, double a, int dirmask, int tt,
                      cudaStream_t s) {
  const int plane = g.xh * g.L[1];   // sites of one (z, t) plane of a parity
  if (plane % S != 0 || tt <= 0 || g.L[3] % tt != 0) tt = 0;   // tiled order needs whole blocks and slabs
  const int nyb = plane / S;
  const size_t smem = sizeof(float2) * 72 * S + (epi_has_clover(EPI) ? sizeof(float4) * 18 * S : 0);
  auto kern = k_dslash_mrhs_smem<EPI, S, NQ, MINB>;
  static std::atomic<unsigned> attr_set{0u};   // devices on which this instantiation may take `smem` bytes
  int dev = 0;
  MG_CUDA(cudaGetDevice(&dev));
  if (dev >= 32 || !(attr_set.load() & (1u << dev))) {
    MG_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    if (dev < 32) attr_set.fetch_or(1u << dev);
  }
  kern<<<(unsigned)((g.Vh + S - 1) / S), S * NQ, smem, s>>>(g, parity, nrhs, stride, out, in, gauge, clov, x, (float)a,
                                                           dirmask, nyb, tt);
  MG_LAUNCH();
}

template <int S, int NQ, int MINB>
void dslash_mrhs_smem(const Geom& g, Epilogue epi, int parity, int nrhs, size_t stride, float* out, const float* in,
                      const float* gauge, const float* clov, const float* x, double a, int dirmask, int tt,
                      cudaStream_t s) {
  switch (epi) {
    case EPI_H: launch_mrhs_smem<EPI_H, S, NQ, MINB>(g, parity, nrhs, stride, out, in, gauge, clov, x, a, dirmask, tt, s); break;
    case EPI_CH: launch_mrhs_smem<EPI_CH, S, NQ, MINB>(g, parity, nrhs, stride, out, in, gauge, clov, x, a, dirmask, tt, s); break;
    case EPI_XPAY: launch_mrhs_smem<EPI_XPAY, S, NQ, MINB>(g, parity, nrhs, stride, out, in, gauge, clov, x, a, dirmask, tt, s); break;
    case EPI_CX_PAY: launch_mrhs_smem<EPI_CX_PAY, S, NQ, MINB>(g, parity, nrhs, stride, out, in, gauge, clov, x, a, dirmask, tt, s); break;
    case EPI_C_XPAY: launch_mrhs_smem<EPI_C_XPAY, S, NQ, MINB>(g, parity, nrhs, stride, out, in, gauge, clov, x, a, dirmask, tt, s); break;
  }
}

template <typename T, int NR, int BS, int MINB = 1>
void dslash_mrhs_cfg(const Geom& g, Epilogue epi, int parity, int nrhs, size_t stride, T* out, const T* in,
                     const T* gauge, const T* clov, const T* x, double a, int dirmask, cudaStream_t s) {
  const dim3 grid((unsigned)(((g.Vh + BS - 1) / BS) * ((nrhs + NR - 1) / NR)));
  switch (epi) {
    case EPI_H: k_dslash_mrhs<T, EPI_H, NR, BS, MINB><<<grid, BS, 0, s>>>(g, parity, nrhs, stride, out, in, gauge, clov, x, (T)a, dirmask); break;
    case EPI_CH: k_dslash_mrhs<T, EPI_CH, NR, BS, MINB><<<grid, BS, 0, s>>>(g, parity, nrhs, stride, out, in, gauge, clov, x, (T)a, dirmask); break;
    case EPI_XPAY: k_dslash_mrhs<T, EPI_XPAY, NR, BS, MINB><<<grid, BS, 0, s>>>(g, parity, nrhs, stride, out, in, gauge, clov, x, (T)a, dirmask); break;
    case EPI_CX_PAY: k_dslash_mrhs<T, EPI_CX_PAY, NR, BS, MINB><<<grid, BS, 0, s>>>(g, parity, nrhs, stride, out, in, gauge, clov, x, (T)a, dirmask); break;
    case EPI_C_XPAY: k_dslash_mrhs<T, EPI_C_XPAY, NR, BS, MINB><<<grid, BS, 0, s>>>(g, parity, nrhs, stride, out, in, gauge, clov, x, (T)a, dirmask); break;
  }
  MG_LAUNCH();
}

// config = NR * 1000 + CTA size (NR right-hand sides per thread; FP32: NR in
// {2, 4}, FP64: NR in {1, 2}) [+ 10000, FP32 only: register cap for more
// resident CTAs, __launch_bounds__ minimum of 4 (NR = 2) or 3 (NR = 4) CTAs of 128], or
// 100000 + NY (rhs in threadIdx.y, NY in {4, 8}), or (FP32 only) 200000 +
// 100 S + NQ [+ 10: tiled CTA order] (links staged in shared memory: S sites
// x NQ rhs lanes per CTA; 203204, 203208, 206404, and 203214, 206414 tiled)
template <typename T>
void dslash_mrhs(const Geom& g, Epilogue epi, int parity, int nrhs, size_t stride, T* out, const T* in,
                 const T* gauge, const T* clov, const T* x, double a, int dirmask, int config, cudaStream_t s) {
  if (nrhs < 1) raise(MG_ERR_ARG, "nrhs must be positive");
  if (config >= 100000 && config < 200000) {
    if (config % 100 == 8)
      dslash_mrhs_y<T, 8>(g, epi, parity, nrhs, stride, out, in, gauge, clov, x, a, dirmask, s);
    else
      dslash_mrhs_y<T, 4>(g, epi, parity, nrhs, stride, out, in, gauge, clov, x, a, dirmask, s);
    return;
  }
  constexpr bool f32 = std::is_same<T, float>::value;
  constexpr int NA = f32 ? 2 : 1, NB = f32 ? 4 : 2;
  if (!f32 && config >= 200000) raise(MG_ERR_ARG, "the shared-memory multi-RHS dslash is FP32 only");
  if constexpr (f32) {
    if (config >= 200000) {   // links (and clover) staged in shared memory once for all rhs
      const int tt = (config / 10) % 10 == 1 ? 8 : 0;   // tiled CTA order, slabs of 8 time slices
      const int base = config - 10 * ((config / 10) % 10);
      if (base == 203208)
        dslash_mrhs_smem<32, 8, 3>(g, epi, parity, nrhs, stride, out, in, gauge, clov, x, a, dirmask, tt, s);
      else if (base == 206404)
        dslash_mrhs_smem<64, 4, 3>(g, epi, parity, nrhs, stride, out, in, gauge, clov, x, a, dirmask, tt, s);
      else
        dslash_mrhs_smem<32, 4, 5>(g, epi, parity, nrhs, stride, out, in, gauge, clov, x, a, dirmask, tt, s);
      return;
    }
    if (config >= 10000) {   // register-capped variants (FP32 only: FP64 would spill), CTA of 128
      if ((config - 10000) / 1000 == 4)
        dslash_mrhs_cfg<T, 4, 128, 3>(g, epi, parity, nrhs, stride, out, in, gauge, clov, x, a, dirmask, s);
      else
        dslash_mrhs_cfg<T, 2, 128, 4>(g, epi, parity, nrhs, stride, out, in, gauge, clov, x, a, dirmask, s);
      return;
    }
  }
  const int nr = config / 1000, bs = config % 1000;
  if (nr == NB) {
    if (bs == 64)
      dslash_mrhs_cfg<T, NB, 64>(g, epi, parity, nrhs, stride, out, in, gauge, clov, x, a, dirmask, s);
    else
      dslash_mrhs_cfg<T, NB, 128>(g, epi, parity, nrhs, stride, out, in, gauge, clov, x, a, dirmask, s);
  } else {
    if (bs == 64)
      dslash_mrhs_cfg<T, NA, 64>(g, epi, parity, nrhs, stride, out, in, gauge, clov, x, a, dirmask, s);
    else
      dslash_mrhs_cfg<T, NA, 128>(g, epi, parity, nrhs, stride, out, in, gauge, clov, x, a, dirmask, s);
  }
}
template void dslash_mrhs<float>(const Geom&, Epilogue, int, int, size_t, float*, const float*, const float*,
                                 const float*, const float*, double, int, int, cudaStream_t);
template void dslash_mrhs<double>(const Geom&, Epilogue, int, int, size_t, double*, const double*, const double*,
                                  const double*, const double*, double, int, int, cudaStream_t);

std::vector<int> dslash_mrhs_configs(bool fp32) {
  return fp32 ? std::vector<int>{2064, 2128, 4064, 4128, 12128, 14128, 100004, 100008, 203204, 203208, 206404, 203214, 206414}
              : std::vector<int>{1064, 1128, 2064, 2128, 100004, 100008};
}
int dslash_mrhs_default(bool fp32) { (void)fp32; return 100004; }

// clover multiply of nrhs vectors (one thread per (site, rhs); the rhs is the
// fastest block index, so the clover lines of a site block are shared in L2)
template <typename T>
__global__ void k_clover_apply_mrhs(Geom g, int nrhs, size_t stride, T* out, const T* __restrict__ in,
                                    const T* __restrict__ clov) {
  const int i = (int)(blockIdx.x / nrhs) * blockDim.x + threadIdx.x, r = (int)(blockIdx.x % nrhs);
  if (i >= g.Vh) return;
  cx<T> x[12], y[12];
  SpinorIO<T>::load(in + (size_t)r * stride, g.Vh, i, x);
  clover_mul<T>(clov, g.Vh, i, x, y);
  SpinorIO<T>::store(out + (size_t)r * stride, g.Vh, i, y);
}

template <typename T>
void clover_apply_mrhs(const Geom& g, int nrhs, size_t stride, T* out, const T* in, const T* clov, cudaStream_t s) {
  const int bs = 128;
  k_clover_apply_mrhs<T><<<(unsigned)(((g.Vh + bs - 1) / bs) * nrhs), bs, 0, s>>>(g, nrhs, stride, out, in, clov);
  MG_LAUNCH();
}
template void clover_apply_mrhs<float>(const Geom&, int, size_t, float*, const float*, const float*, cudaStream_t);
template void clover_apply_mrhs<double>(const Geom&, int, size_t, double*, const double*, const double*, cudaStream_t);

// --------------------------------------------------------------------------- directional terms
// Directional hops of the Galerkin construction, sorted while they are in
// registers: a term that crosses a block face is stored for its own
// projection, all others are added (with the identity-slot vector) into a
// float pair, so a column writes 2 vectors and the faces instead of 8 vectors.
struct GalerkinOut {
  float* W[8];
  float* Sh;
  float* Sl;
  int b[4];
  int split[4];   // the coarse lattice has more than one site in this direction
};

template <int MU, bool FWD>
__device__ __forceinline__ void one_dir(const Geom& g, const GalerkinOut& o, const float* in, const float* gauge,
                                        int par, int i, const int c[4], size_t v, float sh[24], float sl[24]) {
  cx<float> acc[12];
#pragma unroll
  for (int k = 0; k < 12; k++) acc[k] = mkc(0.f, 0.f);
  hop_term<float, MU, FWD>(g, in, gauge, par, i, c, acc);
#pragma unroll
  for (int k = 0; k < 12; k++) acc[k] = -0.5f * acc[k];
  const int l = c[MU] % o.b[MU];
  if (o.split[MU] && (FWD ? l == o.b[MU] - 1 : l == 0)) {
    SpinorIO<float>::store(o.W[MU + (FWD ? 0 : 4)] + v + (size_t)par * 24 * g.Vh, g.Vh, i, acc);
  } else {
#pragma unroll
    for (int k = 0; k < 12; k++) {
      df_acc(sh[2 * k], sl[2 * k], acc[k].re);
      df_acc(sh[2 * k + 1], sl[2 * k + 1], acc[k].im);
    }
  }
}

__global__ void __launch_bounds__(128) k_galerkin_hops(Geom g, GalerkinOut o, const float* __restrict__ u,
                                                       const float* __restrict__ slot,
                                                       const float* __restrict__ gauge, size_t vstride) {
  const int gid = blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= 2 * g.Vh) return;
  const int par = gid / g.Vh, i = gid % g.Vh;
  const size_t v = blockIdx.y * vstride, half = (size_t)24 * g.Vh;
  int c[4];
  cb_coords(g, i, par, c);
  const float* in = u + v + (par ? 0 : half);  // neighbours have the other parity
  cx<float> s[12];
  SpinorIO<float>::load(slot + v + par * half, g.Vh, i, s);
  float sh[24], sl[24];
#pragma unroll
  for (int k = 0; k < 12; k++) {
    sh[2 * k] = s[k].re;
    sh[2 * k + 1] = s[k].im;
    sl[2 * k] = sl[2 * k + 1] = 0.f;
  }
  one_dir<0, true>(g, o, in, gauge, par, i, c, v, sh, sl);
  one_dir<1, true>(g, o, in, gauge, par, i, c, v, sh, sl);
  one_dir<2, true>(g, o, in, gauge, par, i, c, v, sh, sl);
  one_dir<3, true>(g, o, in, gauge, par, i, c, v, sh, sl);
  one_dir<0, false>(g, o, in, gauge, par, i, c, v, sh, sl);
  one_dir<1, false>(g, o, in, gauge, par, i, c, v, sh, sl);
  one_dir<2, false>(g, o, in, gauge, par, i, c, v, sh, sl);
  one_dir<3, false>(g, o, in, gauge, par, i, c, v, sh, sl);
#pragma unroll
  for (int k = 0; k < 12; k++) s[k] = mkc(sh[2 * k], sh[2 * k + 1]);
  SpinorIO<float>::store(o.Sh + v + par * half, g.Vh, i, s);
#pragma unroll
  for (int k = 0; k < 12; k++) s[k] = mkc(sl[2 * k], sl[2 * k + 1]);
  SpinorIO<float>::store(o.Sl + v + par * half, g.Vh, i, s);
}

void galerkin_hops(const Geom& g, const int block[4], const int cdims[4], const float* u, const float* slot,
                   float* const W[8], float* Sh, float* Sl, size_t vstride, int ncol, const float* gauge,
                   cudaStream_t s) {
  GalerkinOut o;
  for (int d = 0; d < 8; d++) o.W[d] = W[d];
  o.Sh = Sh;
  o.Sl = Sl;
  for (int m = 0; m < 4; m++) {
    o.b[m] = block[m];
    o.split[m] = cdims[m] > 1;
  }
  const int n = 2 * g.Vh, bs = 128;
  k_galerkin_hops<<<dim3((n + bs - 1) / bs, ncol), bs, 0, s>>>(g, o, u, slot, gauge, vstride);
  MG_LAUNCH();
}

// --------------------------------------------------------------------------- Philox start vectors
__global__ void k_philox_fine(Geom g, uint64_t seed, int level, int k, float* even, float* odd) {
  const int lex = blockIdx.x * blockDim.x + threadIdx.x;
  if (lex >= 2 * g.Vh) return;
  int c[4];
  int r = lex;
  c[0] = r % g.L[0]; r /= g.L[0];
  c[1] = r % g.L[1]; r /= g.L[1];
  c[2] = r % g.L[2]; c[3] = r / g.L[2];
  const int par = (c[0] + c[1] + c[2] + c[3]) & 1;
  cx<float> s[12];
  for (int d = 0; d < 12; d++) {
    cx<double> z = philox_gauss(seed, level, k, lex, d);
    s[d] = mkc((float)z.re, (float)z.im);
  }
  SpinorIO<float>::store(par ? odd : even, g.Vh, lex >> 1, s);
}

void philox_fine_vector(const Geom& g, uint64_t seed, int level, int k, float* even, float* odd, cudaStream_t s) {
  const int n = 2 * g.Vh, bs = 128;
  k_philox_fine<<<(n + bs - 1) / bs, bs, 0, s>>>(g, seed, level, k, even, odd);
  MG_LAUNCH();
}

}  // namespace mg
