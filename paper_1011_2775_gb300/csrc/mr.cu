// Minimal-residual smoothing on the fine level, fused (section "Adaptive
// multigrid": the cycle's smoother; FP32, like the rest of the cycle).
//
// One MR step on D_r y = y - H_eo A_o^{-1} H_oe A_e^{-1} y with residual r:
//   w = D_r r,  alpha = <w, r> / <w, w>,  e += alpha r,  r -= alpha w.
// The unfused step runs five kernels (clover apply, two dslash, the two-dot
// reduction, the update).  Here it runs three:
//   k_dslash<EPI_CH>               t_o = A_o^{-1} H_oe s_e       (s_e = A_e^{-1} r_e)
//   k_mr_dslash_dot                w_e = r_e - H_eo t_o, and <w, w>, <w, r>
//   k_mr_update_clover             e += alpha r, r -= alpha w, s_e = A_e^{-1} r_e
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
// <w, r> = sum conj(w) r.  One site per thread in CTAs of BS sites (site_block;
// grid-stride only where the partial sums would not fit): with 256 threads and
// 96 registers two CTAs fitted an SM and 331776 sites took 96 us, 77.5 us with
// FP64 sums at 80 registers.
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

// e += alpha r, r -= alpha w (alpha = in[1..2] / in[0]), and s = A_e^{-1} r
// of the updated r on even sites
__global__ void __launch_bounds__(128) k_mr_update_clover(Geom g, float* __restrict__ e, float* __restrict__ r,
                                                          const float* __restrict__ w, const double* __restrict__ in,
                                                          const float* __restrict__ clov, float* __restrict__ s) {
  __shared__ float s_al[2];   // two FP64 divisions per block, not per thread
  if (threadIdx.x < 2) s_al[threadIdx.x] = (float)(in[1 + threadIdx.x] / (in[0] > 0 ? in[0] : 1.0));
  __syncthreads();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.Vh) return;
  const float ar = s_al[0], ai = s_al[1];
  cx<float> ev[12], rv[12], wv[12], sv[12];
  SpinorIO<float>::load(e, g.Vh, i, ev);
  SpinorIO<float>::load(r, g.Vh, i, rv);
  SpinorIO<float>::load(w, g.Vh, i, wv);
#pragma unroll
  for (int k = 0; k < 12; k++) {
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

}  // namespace

void mr_smooth_fine(Ctx* c, float* e, float* r, float* w, float* s, float* t, int nu, double* d_scr) {
  const Geom& g = c->g;
  const size_t n = 12 * c->Vh;
  cudaStream_t st = c->stream;
  blas_zero<float>(e, n, st);
  if (nu <= 0) return;
  clover_apply<float>(g, s, r, c->Ainv<float>(0), st);   // s_e = A_e^{-1} r_e
  const int bs = site_block(c->Vh);
  const long long most = Workspace::kMaxBlocks * (long long)Workspace::kMaxResults / 3;   // three partial sums per CTA
  const unsigned grid_dot = (unsigned)std::min<long long>(most, ((long long)c->Vh + bs - 1) / bs);
  auto dslash_dot = [&]() {
    double* part = c->ws.partials.as<double>();
    unsigned* cnt = c->ws.counter.as<unsigned>();
    const float* U = c->gauge<float>();
    if (bs == 128)
      k_mr_dslash_dot<128><<<grid_dot, 128, 0, st>>>(g, w, t, U, r, part, cnt, d_scr);
    else if (bs == 64)
      k_mr_dslash_dot<64><<<grid_dot, 64, 0, st>>>(g, w, t, U, r, part, cnt, d_scr);
    else
      k_mr_dslash_dot<32><<<grid_dot, 32, 0, st>>>(g, w, t, U, r, part, cnt, d_scr);
    MG_LAUNCH();
  };
  for (int it = 0; it < nu; it++) {
    dslash<float>(g, EPI_CH, 1, t, s, c->gauge<float>(), c->Ainv<float>(1), nullptr, 0.0, 0xff, st);
    dslash_dot();
    c->dslash_launches += 2;
    if (it + 1 < nu) {
      k_mr_update_clover<<<(c->Vh + bs - 1) / bs, bs, 0, st>>>(g, e, r, w, d_scr, c->Ainv<float>(0), s);
      MG_LAUNCH();
    } else {
      blas_mr_update<float>(e, r, w, d_scr, n, st);
    }
  }
}

}  // namespace mg
