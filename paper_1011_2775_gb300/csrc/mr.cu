// Minimal-residual smoothing on the fine level, fused (section "Adaptive
// multigrid": the cycle's smoother; FP32, like the rest of the cycle).
//
// The post-smoothing z += MR_nu(b - D_r z) starts from the residual r = b - D_r z
// of D_r y = y - H_eo A_o^{-1} H_oe A_e^{-1} y and takes nu steps
//   w = D_r r,  alpha = <w, r> / <w, w>,  e += alpha r,  r -= alpha w,   then z += e.
// Unfused, the residual takes five passes and a step five kernels (clover
// apply, two dslash, the two-dot reduction, the update).  Here:
//   k_mr_residual                  r_e = b_e - z_e + H_eo t_o, s_e = A_e^{-1} r_e
//   k_dslash<EPI_CH>               t_o = A_o^{-1} H_oe s_e       (s_e = A_e^{-1} r_e)
//   k_mr_dslash_dot                w_e = r_e - H_eo t_o, and <w, w>, <w, r>
//   k_mr_update_clover             e += alpha r, r -= alpha w, s_e = A_e^{-1} r_e
//   k_mr_finish                    z += e + alpha r (last step; its r is not needed)
// The clover product A_e^{-1} r of the next step is taken from the update
// (site-local), and the two inner products from the dslash epilogue (w and r
// are in registers there).  Sums: FP32 per site (12 components), double-float
// across the sites of a block, FP64 across blocks, in a fixed order, so the
// result does not depend on block scheduling.
#include "dfloat.cuh"
#include "internal.h"
#include "wilson_dev.cuh"

namespace mg {
namespace {


// w_e = r_e - H_eo t_o on even sites, with out[0] = <w, w>, out[1] + i out[2] =
// <w, r> = sum conj(w) r.  One site per thread in CTAs of BS sites (128 or 64;
// grid-stride only where the partial sums would not fit): with 256 threads and
// 96 registers two CTAs fitted an SM and 331776 sites took 96 us, 60 us here.
// CTAs of 32 leave the last one too many partial sums: 49152 sites took 17.3 us,
// 65536 sites in CTAs of 64 14.0 us.
template <int BS>
__global__ void __launch_bounds__(BS, 640 / BS) k_mr_dslash_dot(Geom g, float* __restrict__ w, const float* __restrict__ t,
                                                              const float* __restrict__ gauge,
                                                              const float* __restrict__ r, double* partials,
                                                              unsigned* counter, double* out) {
  df s0 = df_of(0.f), s1 = df_of(0.f), s2 = df_of(0.f);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.Vh; i += gridDim.x * blockDim.x) {
    int c[4];
    cb_coords(g, i, 0, c);
    cx<float> acc[12];
#pragma unroll
    for (int k = 0; k < 12; k++) acc[k] = mkc<float>(0.f, 0.f);
    hop_sum<float>(g, t, gauge, 0, i, c, 0xff, acc);
    cx<float> rv[12], wv[12];
    SpinorIO<float>::load(r, g.Vh, i, rv);
    float a0 = 0.f, a1 = 0.f, a2 = 0.f;
#pragma unroll
    for (int k = 0; k < 12; k++) {
      // r - H_eo t with H = -1/2 sum (1 -+ gamma) U shift: r + acc / 2
      wv[k] = mkc(rv[k].re + 0.5f * acc[k].re, rv[k].im + 0.5f * acc[k].im);
      a0 = fmaf(wv[k].re, wv[k].re, fmaf(wv[k].im, wv[k].im, a0));
      a1 = fmaf(wv[k].re, rv[k].re, fmaf(wv[k].im, rv[k].im, a1));
      a2 = fmaf(wv[k].re, rv[k].im, fmaf(-wv[k].im, rv[k].re, a2));
    }
    SpinorIO<float>::store(w, g.Vh, i, wv);
    s0 = df_add(s0, df_of(a0));
    s1 = df_add(s1, df_of(a1));
    s2 = df_add(s2, df_of(a2));
  }
  const df v[3] = {s0, s1, s2};
  grid_sum<BS, 3>(v, partials, counter, out);
}

// The same with four lanes per site (wilson_dev.cuh), for small lattices (8.0 ->
// 6.4 us at 4096 sites): CTAs of 128 threads, since every CTA is a partial sum
// for the last one to add (8.6 us in CTAs of 32).
__global__ void __launch_bounds__(128) k_mr_dslash_dot_lanes(Geom g, float* __restrict__ w,
                                                             const float* __restrict__ t,
                                                             const float* __restrict__ gauge,
                                                             const float* __restrict__ r, double* partials,
                                                             unsigned* counter, double* out) {
  const int l = blockIdx.x * 128 + threadIdx.x;
  const int k = l & 1, b = (l >> 1) & 1, sp = 2 * b + k;
  const bool live = (l >> 2) < g.Vh;
  const int i = live ? l >> 2 : g.Vh - 1;
  cx<float> acc[3];
  lane_hop_sum<float>(g, t, gauge, 0, i, k, b, acc);
  float v[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int q = 0; q < 3; q++) {
    const cx<float> rv = SpinorIO<float>::get(r, g.Vh, i, 3 * sp + q);
    const cx<float> wv = mkc(rv.re + 0.5f * acc[q].re, rv.im + 0.5f * acc[q].im);
    if (live) {
      v[0] = fmaf(wv.re, wv.re, fmaf(wv.im, wv.im, v[0]));
      v[1] = fmaf(wv.re, rv.re, fmaf(wv.im, rv.im, v[1]));
      v[2] = fmaf(wv.re, rv.im, fmaf(-wv.im, rv.re, v[2]));
      SpinorIO<float>::put(w, g.Vh, i, 3 * sp + q, wv);
    }
  }
  grid_sum<128, 3>(v, partials, counter, out);
}

// r_e = b_e - z_e + H_eo t_o and s_e = A_e^{-1} r_e
__global__ void __launch_bounds__(128) k_mr_residual(Geom g, float* __restrict__ r, float* __restrict__ s,
                                                     const float* __restrict__ t, const float* __restrict__ gauge,
                                                     const float* __restrict__ z, const float* __restrict__ b,
                                                     const float* __restrict__ clov) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.Vh) return;
  int c[4];
  cb_coords(g, i, 0, c);
  cx<float> acc[12], zv[12], bv[12], sv[12];
#pragma unroll
  for (int k = 0; k < 12; k++) acc[k] = mkc<float>(0.f, 0.f);
  hop_sum<float>(g, t, gauge, 0, i, c, 0xff, acc);
  SpinorIO<float>::load(z, g.Vh, i, zv);
  SpinorIO<float>::load(b, g.Vh, i, bv);
#pragma unroll
  for (int k = 0; k < 12; k++)
    bv[k] = mkc(bv[k].re - (zv[k].re + 0.5f * acc[k].re), bv[k].im - (zv[k].im + 0.5f * acc[k].im));
  SpinorIO<float>::store(r, g.Vh, i, bv);
  clover_mul<float>(clov, g.Vh, i, bv, sv);
  SpinorIO<float>::store(s, g.Vh, i, sv);
}

__global__ void __launch_bounds__(128) k_mr_residual_lanes(Geom g, float* __restrict__ r, float* __restrict__ s,
                                                           const float* __restrict__ t, const float* __restrict__ gauge,
                                                           const float* __restrict__ z, const float* __restrict__ bb,
                                                           const float* __restrict__ clov) {
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  const int k = l & 1, b = (l >> 1) & 1, sp = 2 * b + k;
  const bool live = (l >> 2) < g.Vh;
  const int i = live ? l >> 2 : g.Vh - 1;
  cx<float> acc[3], rv[3], sv[3];
  lane_hop_sum<float>(g, t, gauge, 0, i, k, b, acc);
#pragma unroll
  for (int q = 0; q < 3; q++) {
    const cx<float> zv = SpinorIO<float>::get(z, g.Vh, i, 3 * sp + q), bv = SpinorIO<float>::get(bb, g.Vh, i, 3 * sp + q);
    rv[q] = mkc(bv.re - (zv.re + 0.5f * acc[q].re), bv.im - (zv.im + 0.5f * acc[q].im));
  }
  lane_clover<float>(clov, g.Vh, i, k, b, rv, sv);
  if (!live) return;
#pragma unroll
  for (int q = 0; q < 3; q++) {
    SpinorIO<float>::put(r, g.Vh, i, 3 * sp + q, rv[q]);
    SpinorIO<float>::put(s, g.Vh, i, 3 * sp + q, sv[q]);
  }
}

// e += alpha r (e = alpha r on the first step), r -= alpha w (alpha = in[1..2] /
// in[0]), and s = A_e^{-1} r of the updated r on even sites; nrhs right-hand
// sides `stride` floats apart (scalars four apart), neighbouring CTAs sharing
// the sites and so the clover matrices
template <bool FIRST>
__global__ void __launch_bounds__(128) k_mr_update_clover(Geom g, float* __restrict__ e, float* __restrict__ r,
                                                          const float* __restrict__ w, const double* __restrict__ in,
                                                          const float* __restrict__ clov, float* __restrict__ s,
                                                          int nrhs, size_t stride) {
  __shared__ float s_al[2];   // two FP64 divisions per block, not per thread
  const int q = blockIdx.x % nrhs;
  in += 4 * q;
  if (threadIdx.x < 2) s_al[threadIdx.x] = (float)(in[1 + threadIdx.x] / (in[0] > 0 ? in[0] : 1.0));
  __syncthreads();
  const int i = (blockIdx.x / nrhs) * blockDim.x + threadIdx.x;
  e += q * stride;
  r += q * stride;
  w += q * stride;
  s += q * stride;
  if (i >= g.Vh) return;
  const float ar = s_al[0], ai = s_al[1];
  cx<float> ev[12], rv[12], wv[12], sv[12];
  if (!FIRST) SpinorIO<float>::load(e, g.Vh, i, ev);
  SpinorIO<float>::load(r, g.Vh, i, rv);
  SpinorIO<float>::load(w, g.Vh, i, wv);
#pragma unroll
  for (int k = 0; k < 12; k++) {
    if (FIRST) ev[k] = mkc(0.f, 0.f);
    ev[k].re += ar * rv[k].re - ai * rv[k].im;
    ev[k].im += ar * rv[k].im + ai * rv[k].re;
    rv[k].re -= ar * wv[k].re - ai * wv[k].im;
    rv[k].im -= ar * wv[k].im + ai * wv[k].re;
  }
  SpinorIO<float>::store(e, g.Vh, i, ev);
  SpinorIO<float>::store(r, g.Vh, i, rv);
  clover_mul<float>(clov, g.Vh, i, rv, sv);
  SpinorIO<float>::store(s, g.Vh, i, sv);
}

// z += e + alpha r (without e when FIRST), pairs of complex numbers; blockIdx.y:
// right-hand side (packed vectors)
template <bool FIRST>
__global__ void __launch_bounds__(256) k_mr_finish(float4* __restrict__ z, const float4* __restrict__ e,
                                                   const float4* __restrict__ r, const double* __restrict__ in, int n2) {
  __shared__ float s_al[2];
  in += 4 * blockIdx.y;
  z += (size_t)blockIdx.y * n2;
  e += (size_t)blockIdx.y * n2;
  r += (size_t)blockIdx.y * n2;
  if (threadIdx.x < 2) s_al[threadIdx.x] = (float)(in[1 + threadIdx.x] / (in[0] > 0 ? in[0] : 1.0));
  __syncthreads();
  const float ar = s_al[0], ai = s_al[1];
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n2; i += gridDim.x * blockDim.x) {
    const float4 rv = r[i];
    float4 zv = z[i];
    float4 ev = make_float4(0.f, 0.f, 0.f, 0.f);
    if (!FIRST) ev = e[i];
    ev.x += ar * rv.x - ai * rv.y;
    ev.y += ar * rv.y + ai * rv.x;
    ev.z += ar * rv.z - ai * rv.w;
    ev.w += ar * rv.w + ai * rv.z;
    z[i] = make_float4(zv.x + ev.x, zv.y + ev.y, zv.z + ev.z, zv.w + ev.w);
  }
}

// s = A_e^{-1} z and d = b - z for nrhs right-hand sides
__global__ void __launch_bounds__(128) k_mr_begin(Geom g, float* __restrict__ s, float* __restrict__ d,
                                                  const float* __restrict__ z, const float* __restrict__ b,
                                                  const float* __restrict__ clov, int nrhs, size_t stride) {
  const int q = blockIdx.x % nrhs, i = (blockIdx.x / nrhs) * blockDim.x + threadIdx.x;
  if (i >= g.Vh) return;
  const size_t o = q * stride;
  cx<float> zv[12], bv[12], sv[12];
  SpinorIO<float>::load(z + o, g.Vh, i, zv);
  SpinorIO<float>::load(b + o, g.Vh, i, bv);
#pragma unroll
  for (int k = 0; k < 12; k++) bv[k] = mkc(bv[k].re - zv[k].re, bv[k].im - zv[k].im);
  SpinorIO<float>::store(d + o, g.Vh, i, bv);
  clover_mul<float>(clov, g.Vh, i, zv, sv);
  SpinorIO<float>::store(s + o, g.Vh, i, sv);
}

}  // namespace

void mr_post_smooth_fine(Ctx* c, float* z, const float* b, float* e, float* r, float* w, float* s, float* t, int nu,
                         double* d_scr) {
  const Geom& g = c->g;
  cudaStream_t st = c->stream;
  if (nu <= 0) return;
  const float* U = c->gauge<float>();
  const int bs = site_block(c->Vh);
  const unsigned sites = (unsigned)((c->Vh + bs - 1) / bs);
  // four lanes per site by the rule of the dslash; partial sums: three per CTA
  const bool lanes = dslash_lanes_f32(g.Vh);
  const int bl = site_block(4 * (long long)c->Vh);
  const unsigned grid_l = (unsigned)((4 * c->Vh + bl - 1) / bl);
  const long long most = Workspace::kMaxBlocks * (long long)Workspace::kMaxResults / 3;
  const unsigned grid_dot = (unsigned)std::min<long long>(most, bs == 128 ? sites : (c->Vh + 63) / 64);
  double* part = c->ws.partials.as<double>();
  unsigned* cnt = c->ws.counter.as<unsigned>();
  auto dslash_dot = [&]() {
    if (lanes) {
      k_mr_dslash_dot_lanes<<<(unsigned)((4 * c->Vh + 127) / 128), 128, 0, st>>>(g, w, t, U, r, part, cnt, d_scr);
    } else if (bs == 128) {
      k_mr_dslash_dot<128><<<grid_dot, 128, 0, st>>>(g, w, t, U, r, part, cnt, d_scr);
    } else {
      k_mr_dslash_dot<64><<<grid_dot, 64, 0, st>>>(g, w, t, U, r, part, cnt, d_scr);
    }
    MG_LAUNCH();
  };
  auto half_dr = [&]() {   // t_o = A_o^{-1} H_oe s_e
    dslash<float>(g, EPI_CH, 1, t, s, U, c->Ainv<float>(1), nullptr, 0.0, 0xff, st);
    c->dslash_launches += 2;
  };
  clover_apply<float>(g, s, z, c->Ainv<float>(0), st);
  half_dr();
  if (lanes)
    k_mr_residual_lanes<<<grid_l, bl, 0, st>>>(g, r, s, t, U, z, b, c->Ainv<float>(0));
  else
    k_mr_residual<<<sites, bs, 0, st>>>(g, r, s, t, U, z, b, c->Ainv<float>(0));
  MG_LAUNCH();
  for (int it = 0; it < nu; it++) {
    half_dr();
    dslash_dot();
    if (it + 1 < nu) {
      if (it == 0)
        k_mr_update_clover<true><<<sites, bs, 0, st>>>(g, e, r, w, d_scr, c->Ainv<float>(0), s, 1, 0);
      else
        k_mr_update_clover<false><<<sites, bs, 0, st>>>(g, e, r, w, d_scr, c->Ainv<float>(0), s, 1, 0);
    } else {
      const int n2 = (int)(6 * c->Vh), grid = (int)std::min<long long>(152 * 8, (n2 + 255) / 256);
      if (it == 0)
        k_mr_finish<true><<<grid, 256, 0, st>>>((float4*)z, (const float4*)e, (const float4*)r, d_scr, n2);
      else
        k_mr_finish<false><<<grid, 256, 0, st>>>((float4*)z, (const float4*)e, (const float4*)r, d_scr, n2);
    }
    MG_LAUNCH();
  }
}

// The same for nb right-hand sides (packed half vectors) with the multi-RHS
// hops: d = b - z and s = A^{-1} z in one pass, r = d + H t, then per step the hops, the inner
// products, and one pass for e, r and the next A^{-1} r.  The passes run at the
// memory's rate, so what counts is what they do not read and write again.
void mr_post_smooth_multi(Ctx* c, FineOps<float>& F, float* z, const float* b, float* e, float* r, float* w, int nu,
                          int nb, double* d_scr) {
  const Geom& g = c->g;
  cudaStream_t st = c->stream;
  if (nu <= 0) return;
  F.reserve_multi(nb);
  const size_t hs = 24 * (size_t)c->Vh;
  const int bs = site_block((long long)c->Vh * nb);
  const unsigned grid = (unsigned)((c->Vh + bs - 1) / bs) * nb;
  float* s = F.m1.as<float>();
  k_mr_begin<<<grid, bs, 0, st>>>(g, s, w, z, b, c->Ainv<float>(0), nb, hs);
  MG_LAUNCH();
  F.hops_multi(r, w, 1.0, nb);
  clover_apply_mrhs<float>(g, nb, hs, s, r, c->Ainv<float>(0), st);
  for (int it = 0; it < nu; it++) {
    F.hops_multi(w, r, -1.0, nb);
    blas_dot2_multi<float>(w, r, hs / 2, hs, nb, d_scr, c->ws, st);
    if (it + 1 < nu) {
      if (it == 0)
        k_mr_update_clover<true><<<grid, bs, 0, st>>>(g, e, r, w, d_scr, c->Ainv<float>(0), s, nb, hs);
      else
        k_mr_update_clover<false><<<grid, bs, 0, st>>>(g, e, r, w, d_scr, c->Ainv<float>(0), s, nb, hs);
    } else {
      const int n2 = (int)(6 * c->Vh);
      const dim3 gf((unsigned)std::min<long long>((152 * 16 + nb - 1) / nb, (n2 + 255) / 256), nb);
      if (it == 0)
        k_mr_finish<true><<<gf, 256, 0, st>>>((float4*)z, (const float4*)e, (const float4*)r, d_scr, n2);
      else
        k_mr_finish<false><<<gf, 256, 0, st>>>((float4*)z, (const float4*)e, (const float4*)r, d_scr, n2);
    }
    MG_LAUNCH();
  }
}

}  // namespace mg
