// BLAS-1 kernels and deterministic reductions for the GCR solvers
// (section "Adaptive multigrid": GCR is the outer solver; section
// "Implementation": GCR again on every coarse level).
//
// Inner products of FP64 vectors accumulate in FP64; of FP32 vectors in FP32 over
// the few elements of a thread and in double-float across threads.
// Reductions are deterministic: a fixed grid (a function of n only), per-block
// partials written to the workspace, and an ordered final sum by the last
// block to finish (grid_sum in dfloat.cuh).  The GCR kernels fuse the
// orthogonalisation update with the norms it needs and read their
// coefficients from device memory, so a GCR iteration needs no host round
// trip except the optional convergence check.
#include "dfloat.cuh"
#include "internal.h"

namespace mg {

namespace {
constexpr int kBS = 256;

inline int red_grid(size_t n) {
  size_t b = (n + kBS - 1) / kBS;
  if (b < 1) b = 1;
  if (b > (size_t)Workspace::kMaxBlocks) b = Workspace::kMaxBlocks;
  return (int)b;
}
inline int ew_grid(size_t n) {
  size_t b = (n + kBS - 1) / kBS;
  if (b < 1) b = 1;
  if (b > 152 * 16) b = 152 * 16;
  return (int)b;
}

// the grid's sums of NR per-thread values (see grid_sum)
template <int NR, typename T>
__device__ __forceinline__ void grid_reduce(const T (&v)[NR], double* partials, unsigned* counter, double* out) {
  grid_sum<kBS, NR>(v, partials, counter, out);
}

// K complex coefficients read from FP64 device scalars, times `scale`: one
// thread per value converts, all threads read them from shared memory (a
// conversion per thread would queue on the FP64 pipe).
template <int K>
struct Coefs {
  float h[2 * (K > 0 ? K : 1)], l[2 * (K > 0 ? K : 1)];
};
template <int K>
__device__ __forceinline__ void load_coefs(Coefs<K>& s, const double* __restrict__ c, double scale) {
  if (threadIdx.x < 2 * K) {
    const double v = scale * c[threadIdx.x];
    const float h = (float)v;
    s.h[threadIdx.x] = h;
    s.l[threadIdx.x] = (float)(v - (double)h);
  }
  __syncthreads();
}

template <typename T>
struct VecPtrs {
  const cx<T>* p[8];
};

// Per-thread accumulation type: a thread sums only its few grid-stride
// elements, in the vectors' own precision.  Across the threads of a block FP64
// sums are added in FP64 and FP32 sums as float pairs (about 48 bits; in FP64
// where the pairs leave FP32's range), across blocks in FP64 (grid_sum).  On
// GB300 this keeps the FP32 reductions off the (slow) FP64 pipe.
template <typename T>
using acc_t = typename std::conditional<sizeof(T) == 4, float, double>::type;
}  // namespace

// --------------------------------------------------------------------------- elementwise
template <typename T>
__global__ void k_zero(cx<T>* x, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    x[i] = mkc<T>(0, 0);
}
template <typename T>
void blas_zero(T* x, size_t n, cudaStream_t s) {
  k_zero<T><<<ew_grid(n), kBS, 0, s>>>((cx<T>*)x, n);
  MG_LAUNCH();
}

template <typename TI, typename TO>
__global__ void k_convert(cx<TO>* y, const cx<TI>* __restrict__ x, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    y[i] = mkc<TO>((TO)x[i].re, (TO)x[i].im);
}
template <typename TI, typename TO>
void blas_convert(TO* y, const TI* x, size_t n, cudaStream_t s) {
  k_convert<TI, TO><<<ew_grid(n), kBS, 0, s>>>((cx<TO>*)y, (const cx<TI>*)x, n);
  MG_LAUNCH();
}

template <typename T>
__global__ void k_axpby(T a, const cx<T>* __restrict__ x, T b, cx<T>* y, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    cx<T> xv = x[i], yv = y[i];
    y[i] = mkc<T>(a * xv.re + b * yv.re, a * xv.im + b * yv.im);
  }
}
template <typename T>
void blas_axpby(double a, const T* x, double b, T* y, size_t n, cudaStream_t s) {
  k_axpby<T><<<ew_grid(n), kBS, 0, s>>>((T)a, (const cx<T>*)x, (T)b, (cx<T>*)y, n);
  MG_LAUNCH();
}

// --------------------------------------------------------------------------- reductions
template <typename T>
__global__ void k_norm2(const cx<T>* __restrict__ x, size_t n, double* partials, unsigned* counter, double* out) {
  acc_t<T> s = 0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    cx<T> a = x[i];
    s = fma((acc_t<T>)a.re, (acc_t<T>)a.re, s);
    s = fma((acc_t<T>)a.im, (acc_t<T>)a.im, s);
  }
  const acc_t<T> v[1] = {s};
  grid_reduce<1>(v, partials, counter, out);
}
template <typename T>
void blas_norm2(const T* x, size_t n, double* d_out, Workspace& ws, cudaStream_t s) {
  k_norm2<T><<<red_grid(n), kBS, 0, s>>>((const cx<T>*)x, n, ws.partials.as<double>(), ws.counter.as<unsigned>(), d_out);
  MG_LAUNCH();
}

template <typename T>
__global__ void k_cdot(const cx<T>* __restrict__ x, const cx<T>* __restrict__ y, size_t n, double* partials,
                       unsigned* counter, double* out) {
  acc_t<T> s0 = 0, s1 = 0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    cx<T> a = x[i], b = y[i];
    s0 = fma((acc_t<T>)a.re, (acc_t<T>)b.re, s0);
    s0 = fma((acc_t<T>)a.im, (acc_t<T>)b.im, s0);
    s1 = fma((acc_t<T>)a.re, (acc_t<T>)b.im, s1);
    s1 = fma(-(acc_t<T>)a.im, (acc_t<T>)b.re, s1);
  }
  const acc_t<T> v[2] = {s0, s1};
  grid_reduce<2>(v, partials, counter, out);
}
template <typename T>
void blas_cdot(const T* x, const T* y, size_t n, double* d_out, Workspace& ws, cudaStream_t s) {
  k_cdot<T><<<red_grid(n), kBS, 0, s>>>((const cx<T>*)x, (const cx<T>*)y, n, ws.partials.as<double>(),
                                        ws.counter.as<unsigned>(), d_out);
  MG_LAUNCH();
}

template <typename T>
__global__ void k_dot2(const cx<T>* __restrict__ w, const cx<T>* __restrict__ r, size_t n, double* partials,
                       unsigned* counter, double* out) {
  acc_t<T> s0 = 0, s1 = 0, s2 = 0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    cx<T> a = w[i], b = r[i];
    s0 = fma((acc_t<T>)a.re, (acc_t<T>)a.re, s0);
    s0 = fma((acc_t<T>)a.im, (acc_t<T>)a.im, s0);
    s1 = fma((acc_t<T>)a.re, (acc_t<T>)b.re, s1);
    s1 = fma((acc_t<T>)a.im, (acc_t<T>)b.im, s1);
    s2 = fma((acc_t<T>)a.re, (acc_t<T>)b.im, s2);
    s2 = fma(-(acc_t<T>)a.im, (acc_t<T>)b.re, s2);
  }
  const acc_t<T> v[3] = {s0, s1, s2};
  grid_reduce<3>(v, partials, counter, out);
}
// nrhs pairs (w_q, r_q) of FP32 vectors at `stride` floats apart: d_out[4q ..
// 4q+2] per pair, one launch (blockIdx.y = q, a separate reduction per pair);
// 16 bytes per load (n is even).  With many pairs a thread has many elements, so
// its running sums are float pairs: the FP32 part of a sum is the two products of
// one complex number.
__global__ void __launch_bounds__(kBS) k_dot2_multi(const float* __restrict__ w, const float* __restrict__ r, size_t n2,
                                                    size_t stride, double* partials, unsigned* counters, double* out) {
  const int q = blockIdx.y;
  const float4* w4 = reinterpret_cast<const float4*>(w + q * stride);
  const float4* r4 = reinterpret_cast<const float4*>(r + q * stride);
  float h[3] = {}, l[3] = {};
#pragma unroll 4
  for (size_t i = blockIdx.x * (size_t)kBS + threadIdx.x; i < n2; i += (size_t)gridDim.x * kBS) {
    const float4 a = w4[i], b = r4[i];
    df_acc(h[0], l[0], fmaf(a.x, a.x, a.y * a.y));
    df_acc(h[1], l[1], fmaf(a.x, b.x, a.y * b.y));
    df_acc(h[2], l[2], fmaf(a.x, b.y, -a.y * b.x));
    df_acc(h[0], l[0], fmaf(a.z, a.z, a.w * a.w));
    df_acc(h[1], l[1], fmaf(a.z, b.z, a.w * b.w));
    df_acc(h[2], l[2], fmaf(a.z, b.w, -a.w * b.z));
  }
  df v[3];
#pragma unroll
  for (int k = 0; k < 3; k++) v[k] = df_norm(h[k], l[k]);
  grid_reduce<3>(v, partials + (size_t)q * gridDim.x * 3, counters + q, out + 4 * q);
}
template <typename T>
void blas_dot2_multi(const T* w, const T* r, size_t n, size_t stride, int nrhs, double* d_out, Workspace& ws,
                     cudaStream_t s) {
  if (nrhs > Workspace::kMultiCounters) raise(MG_ERR_ARG, "too many vectors for one multi-reduction");
  // a wave of CTAs over all pairs: every CTA is a partial sum for the last one of its pair to add
  const int g = std::max(1, std::min(red_grid(n / 2), 152 * 8 / nrhs));
  k_dot2_multi<<<dim3(g, nrhs), kBS, 0, s>>>(w, r, n / 2, stride, ws.partials.as<double>(), ws.mcounters.as<unsigned>(),
                                             d_out);
  MG_LAUNCH();
}

template <typename T>
__global__ void k_mr_update_multi(cx<T>* e, cx<T>* r, const cx<T>* __restrict__ w, const double* __restrict__ in,
                                  size_t n, size_t stride) {
  const int q = blockIdx.y;
  e += q * stride;
  r += q * stride;
  w += q * stride;
  in += 4 * q;
  __shared__ T s_al[2];
  if (threadIdx.x < 2) s_al[threadIdx.x] = (T)(in[1 + threadIdx.x] / (in[0] > 0 ? in[0] : 1.0));
  __syncthreads();
  const T ar = s_al[0], ai = s_al[1];
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    cx<T> rv = r[i], wv = w[i], ev = e[i];
    ev.re = fma(ar, rv.re, fma(-ai, rv.im, ev.re));
    ev.im = fma(ar, rv.im, fma(ai, rv.re, ev.im));
    rv.re = fma(-ar, wv.re, fma(ai, wv.im, rv.re));
    rv.im = fma(-ar, wv.im, fma(-ai, wv.re, rv.im));
    e[i] = ev;
    r[i] = rv;
  }
}
template <typename T>
void blas_mr_update_multi(T* e, T* r, const T* w, const double* d_in, size_t n, size_t stride, int nrhs,
                          cudaStream_t s) {
  int g = ew_grid(n);
  if (g * nrhs > 152 * 16) g = (152 * 16 + nrhs - 1) / nrhs;
  k_mr_update_multi<T><<<dim3(g, nrhs), kBS, 0, s>>>((cx<T>*)e, (cx<T>*)r, (const cx<T>*)w, d_in, n, stride / 2);
  MG_LAUNCH();
}
template void blas_dot2_multi<float>(const float*, const float*, size_t, size_t, int, double*, Workspace&, cudaStream_t);
template void blas_mr_update_multi<float>(float*, float*, const float*, const double*, size_t, size_t, int,
                                          cudaStream_t);

template <typename T>
void blas_dot2(const T* w, const T* r, size_t n, double* d_out, Workspace& ws, cudaStream_t s) {
  k_dot2<T><<<red_grid(n), kBS, 0, s>>>((const cx<T>*)w, (const cx<T>*)r, n, ws.partials.as<double>(),
                                        ws.counter.as<unsigned>(), d_out);
  MG_LAUNCH();
}

// d_out[2j..] = <V_j, w>, j < K.  FP64: bound by the FP64 pipe (4 K operations
// per element of 64 cycles per warp), so two CTAs per SM are enough to hide the
// loads and halve the sums over lanes and blocks, which queue on the same pipe.
// FP32: pairs of complex numbers, 16 bytes per load, with a sum for the first
// and one for the second of a pair (n is even: 12 or 2 Nv components a site).
// Eight vectors: FP64, 0.79 M complex, 57.2 -> 52.3 us (40 us of the pipe); FP32,
// 1.57 M complex, 47.5 -> 26.1 us (17 us of memory traffic).
constexpr int kDotGrid64 = 304;
template <int K>
__global__ void __launch_bounds__(kBS) k_multidot_pairs(VecPtrs<float> V, const float4* __restrict__ w, size_t n2,
                                                        double* partials, unsigned* counter, double* out) {
  float s[2][2 * K];
#pragma unroll
  for (int r = 0; r < 2 * K; r++) s[0][r] = s[1][r] = 0.f;
  for (size_t i = blockIdx.x * (size_t)kBS + threadIdx.x; i < n2; i += (size_t)gridDim.x * kBS) {
    float4 a[K];
#pragma unroll
    for (int j = 0; j < K; j++) a[j] = reinterpret_cast<const float4*>(V.p[j])[i];
    const float4 b = w[i];
#pragma unroll
    for (int j = 0; j < K; j++) {
      s[0][2 * j] = fmaf(a[j].x, b.x, fmaf(a[j].y, b.y, s[0][2 * j]));
      s[0][2 * j + 1] = fmaf(a[j].x, b.y, fmaf(-a[j].y, b.x, s[0][2 * j + 1]));
      s[1][2 * j] = fmaf(a[j].z, b.z, fmaf(a[j].w, b.w, s[1][2 * j]));
      s[1][2 * j + 1] = fmaf(a[j].z, b.w, fmaf(-a[j].w, b.z, s[1][2 * j + 1]));
    }
  }
  df v[2 * K];
#pragma unroll
  for (int r = 0; r < 2 * K; r++) v[r] = df_add(df_of(s[0][r]), df_of(s[1][r]));
  grid_reduce<2 * K>(v, partials, counter, out);
}
template <typename T, int K>
__global__ void k_multidot(VecPtrs<T> V, const cx<T>* __restrict__ w, size_t n, double* partials, unsigned* counter,
                           double* out) {
  acc_t<T> s[2 * K];
#pragma unroll
  for (int r = 0; r < 2 * K; r++) s[r] = 0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    cx<T> b = w[i];
#pragma unroll
    for (int j = 0; j < K; j++) {
      cx<T> a = V.p[j][i];
      s[2 * j] = fma((acc_t<T>)a.re, (acc_t<T>)b.re, s[2 * j]);
      s[2 * j] = fma((acc_t<T>)a.im, (acc_t<T>)b.im, s[2 * j]);
      s[2 * j + 1] = fma((acc_t<T>)a.re, (acc_t<T>)b.im, s[2 * j + 1]);
      s[2 * j + 1] = fma(-(acc_t<T>)a.im, (acc_t<T>)b.re, s[2 * j + 1]);
    }
  }
  grid_reduce<2 * K>(s, partials, counter, out);
}

template <typename T>
void blas_multidot(const T* const* V, int k, const T* w, size_t n, double* d_out, Workspace& ws, cudaStream_t s) {
  double* pa = ws.partials.as<double>();
  unsigned* ct = ws.counter.as<unsigned>();
  for (int j0 = 0; j0 < k; j0 += 8) {
    const int kk = (k - j0) < 8 ? (k - j0) : 8;
    VecPtrs<T> P;
    for (int j = 0; j < 8; j++) P.p[j] = (const cx<T>*)(j < kk ? V[j0 + j] : V[j0]);
    double* o = d_out + 2 * j0;
    auto run = [&](auto kc) {
      constexpr int K = decltype(kc)::value;
      if constexpr (sizeof(T) == 4)
        k_multidot_pairs<K><<<red_grid(n / 2), kBS, 0, s>>>(P, (const float4*)w, n / 2, pa, ct, o);
      else
        k_multidot<T, K><<<std::min(red_grid(n), kDotGrid64), kBS, 0, s>>>(P, (const cx<T>*)w, n, pa, ct, o);
    };
    switch (kk) {
      case 1: run(std::integral_constant<int, 1>()); break;
      case 2: run(std::integral_constant<int, 2>()); break;
      case 3: run(std::integral_constant<int, 3>()); break;
      case 4: run(std::integral_constant<int, 4>()); break;
      case 5: run(std::integral_constant<int, 5>()); break;
      case 6: run(std::integral_constant<int, 6>()); break;
      case 7: run(std::integral_constant<int, 7>()); break;
      default: run(std::integral_constant<int, 8>());
    }
    MG_LAUNCH();
  }
}

// w -= sum_{j<K} beta_j V_j; if RED: {||w||^2, <w, r>} -> out.  FP32 vectors in
// pairs of complex numbers (16 bytes per load), as above.
template <int K, bool RED>
__global__ void __launch_bounds__(kBS) k_orth_update_pairs(float4* w, VecPtrs<float> V,
                                                           const double* __restrict__ beta,
                                                           const float4* __restrict__ r, size_t n2, double* partials,
                                                           unsigned* counter, double* out) {
  __shared__ Coefs<K> sb;
  if (K > 0) load_coefs<K>(sb, beta, 1.0);
  float s[2][3] = {};
  for (size_t i = blockIdx.x * (size_t)kBS + threadIdx.x; i < n2; i += (size_t)gridDim.x * kBS) {
    float4 q[K > 0 ? K : 1], b = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int j = 0; j < K; j++) q[j] = reinterpret_cast<const float4*>(V.p[j])[i];
    float4 a = w[i];
    if (RED) b = r[i];
#pragma unroll
    for (int j = 0; j < K; j++) {
      const float br = sb.h[2 * j], bi = sb.h[2 * j + 1];
      a.x = fmaf(-br, q[j].x, fmaf(bi, q[j].y, a.x));
      a.y = fmaf(-br, q[j].y, fmaf(-bi, q[j].x, a.y));
      a.z = fmaf(-br, q[j].z, fmaf(bi, q[j].w, a.z));
      a.w = fmaf(-br, q[j].w, fmaf(-bi, q[j].z, a.w));
    }
    if (K > 0) w[i] = a;
    if (RED) {
      s[0][0] = fmaf(a.x, a.x, fmaf(a.y, a.y, s[0][0]));
      s[0][1] = fmaf(a.x, b.x, fmaf(a.y, b.y, s[0][1]));
      s[0][2] = fmaf(a.x, b.y, fmaf(-a.y, b.x, s[0][2]));
      s[1][0] = fmaf(a.z, a.z, fmaf(a.w, a.w, s[1][0]));
      s[1][1] = fmaf(a.z, b.z, fmaf(a.w, b.w, s[1][1]));
      s[1][2] = fmaf(a.z, b.w, fmaf(-a.w, b.z, s[1][2]));
    }
  }
  df v[3];
#pragma unroll
  for (int q = 0; q < 3; q++) v[q] = df_add(df_of(s[0][q]), df_of(s[1][q]));
  if (RED) grid_reduce<3>(v, partials, counter, out);
}
template <typename T, int K, bool RED>
__global__ void k_orth_update(cx<T>* w, VecPtrs<T> V, const double* __restrict__ beta, const cx<T>* __restrict__ r,
                              size_t n, double* partials, unsigned* counter, double* out) {
  T br[K > 0 ? K : 1], bi[K > 0 ? K : 1];
#pragma unroll
  for (int j = 0; j < K; j++) {
    br[j] = (T)beta[2 * j];
    bi[j] = (T)beta[2 * j + 1];
  }
  acc_t<T> s0 = 0, s1 = 0, s2 = 0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    cx<T> a = w[i];
#pragma unroll
    for (int j = 0; j < K; j++) {
      cx<T> q = V.p[j][i];
      a.re = fma(-br[j], q.re, fma(bi[j], q.im, a.re));   // four operations; written as a -= b q the compiler takes six
      a.im = fma(-br[j], q.im, fma(-bi[j], q.re, a.im));
    }
    if (K > 0) w[i] = a;
    if (RED) {
      cx<T> b = r[i];
      s0 = fma((acc_t<T>)a.re, (acc_t<T>)a.re, s0);
      s0 = fma((acc_t<T>)a.im, (acc_t<T>)a.im, s0);
      s1 = fma((acc_t<T>)a.re, (acc_t<T>)b.re, s1);
      s1 = fma((acc_t<T>)a.im, (acc_t<T>)b.im, s1);
      s2 = fma((acc_t<T>)a.re, (acc_t<T>)b.im, s2);
      s2 = fma(-(acc_t<T>)a.im, (acc_t<T>)b.re, s2);
    }
  }
  const acc_t<T> v[3] = {s0, s1, s2};
  if (RED) grid_reduce<3>(v, partials, counter, out);
}

template <typename T>
void blas_orth_update(T* w, const T* const* V, const double* d_beta, int k, const T* r, size_t n, double* d_out,
                      Workspace& ws, cudaStream_t s) {
  double* pa = ws.partials.as<double>();
  unsigned* ct = ws.counter.as<unsigned>();
  auto launch = [&](auto kc, auto red, const VecPtrs<T>& P, const double* b) {
    constexpr int K = decltype(kc)::value;
    constexpr bool RED = decltype(red)::value;
    if constexpr (sizeof(T) == 4)
      k_orth_update_pairs<K, RED><<<red_grid(n / 2), kBS, 0, s>>>((float4*)w, P, b, (const float4*)r, n / 2, pa, ct, d_out);
    else
      k_orth_update<T, K, RED><<<red_grid(n), kBS, 0, s>>>((cx<T>*)w, P, b, (const cx<T>*)r, n, pa, ct, d_out);
    MG_LAUNCH();
  };
  if (k == 0) {
    launch(std::integral_constant<int, 0>(), std::true_type(), VecPtrs<T>{}, d_beta);
    return;
  }
  for (int j0 = 0; j0 < k; j0 += 8) {
    const int kk = (k - j0) < 8 ? (k - j0) : 8;
    VecPtrs<T> P;
    for (int j = 0; j < 8; j++) P.p[j] = (const cx<T>*)(j < kk ? V[j0 + j] : V[j0]);
    auto run = [&](auto kc) {
      if (j0 + kk >= k)
        launch(kc, std::true_type(), P, d_beta + 2 * j0);
      else
        launch(kc, std::false_type(), P, d_beta + 2 * j0);
    };
    switch (kk) {
      case 1: run(std::integral_constant<int, 1>()); break;
      case 2: run(std::integral_constant<int, 2>()); break;
      case 3: run(std::integral_constant<int, 3>()); break;
      case 4: run(std::integral_constant<int, 4>()); break;
      case 5: run(std::integral_constant<int, 5>()); break;
      case 6: run(std::integral_constant<int, 6>()); break;
      case 7: run(std::integral_constant<int, 7>()); break;
      default: run(std::integral_constant<int, 8>());
    }
  }
}

template <typename T>
__global__ void k_r_update(cx<T>* w, const cx<T>* r, cx<T>* r_out, size_t n, const double* __restrict__ in, double* alpha_out,
                           double* gamma_out, double* partials, unsigned* counter, double* out) {
  // the square root and the divisions by one thread of the block: in every
  // thread they took longer than the pass over the vectors (29.8 us of which
  // about 15 at 0.79 M complex FP64)
  __shared__ T s_ga[3];
  if (threadIdx.x == 0) {
    const double g2 = in[0];
    const double gam = g2 > 0 ? sqrt(g2) : 1.0;
    const double ar = in[1] / gam, ai = in[2] / gam;  // alpha = <w/gamma, r>
    if (blockIdx.x == 0) {
      alpha_out[0] = ar;
      alpha_out[1] = ai;
      gamma_out[0] = gam;
    }
    s_ga[0] = (T)(1.0 / gam);
    s_ga[1] = (T)ar;
    s_ga[2] = (T)ai;
  }
  __syncthreads();
  const T ig = s_ga[0], a_r = s_ga[1], a_i = s_ga[2];
  acc_t<T> s = 0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    cx<T> q = w[i];
    q.re *= ig;
    q.im *= ig;
    w[i] = q;
    cx<T> b = r[i];
    b.re = fma(-a_r, q.re, fma(a_i, q.im, b.re));
    b.im = fma(-a_r, q.im, fma(-a_i, q.re, b.im));
    r_out[i] = b;
    s = fma((acc_t<T>)b.re, (acc_t<T>)b.re, s);
    s = fma((acc_t<T>)b.im, (acc_t<T>)b.im, s);
  }
  const acc_t<T> v[1] = {s};
  grid_reduce<1>(v, partials, counter, out);
}

template <typename T>
void blas_r_update(T* w, const T* r, T* r_out, size_t n, const double* d_in, double* d_alpha, double* d_gamma,
                   double* d_rnorm2,
                   Workspace& ws, cudaStream_t s) {
  k_r_update<T><<<red_grid(n), kBS, 0, s>>>((cx<T>*)w, (const cx<T>*)r, (cx<T>*)r_out, n, d_in, d_alpha, d_gamma, ws.partials.as<double>(),
                                            ws.counter.as<unsigned>(), d_rnorm2);
  MG_LAUNCH();
}

// FP64 results are accumulated in FP64.  FP32 results (FP32 vectors, FP64
// coefficients) are accumulated in compensated FP32 -- about 48 bits before the
// rounding to FP32 -- with the coefficients as float pairs: in FP64 arithmetic
// the pass took ten times its memory time (221 us for eight vectors of 1.57 M
// complex, against 126 MB of traffic).
template <typename T, typename TZ, int K>
__global__ void k_lincomb(cx<T>* x, VecPtrs<TZ> Z, const double* __restrict__ c, double scale, size_t n) {
  if constexpr (sizeof(T) == 4) {   // pairs of complex numbers; n is even
    __shared__ Coefs<K> sc;
    load_coefs<K>(sc, c, scale);
    float4* x4 = reinterpret_cast<float4*>(x);
    const size_t n2 = n / 2;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n2; i += (size_t)gridDim.x * blockDim.x) {
      float4 z[K];
#pragma unroll
      for (int j = 0; j < K; j++) z[j] = reinterpret_cast<const float4*>(Z.p[j])[i];
      const float4 a = x4[i];
      float h[4] = {a.x, a.y, a.z, a.w}, l[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int j = 0; j < K; j++) {
        const float cr = sc.h[2 * j], ci = sc.h[2 * j + 1], lr = sc.l[2 * j], li = sc.l[2 * j + 1];
        const float zr[2] = {z[j].x, z[j].z}, zi[2] = {z[j].y, z[j].w};
#pragma unroll
        for (int u = 0; u < 2; u++) {
          dot2_acc(h[2 * u], l[2 * u], cr, zr[u]);
          dot2_acc(h[2 * u], l[2 * u], -ci, zi[u]);
          l[2 * u] = fmaf(lr, zr[u], fmaf(-li, zi[u], l[2 * u]));
          dot2_acc(h[2 * u + 1], l[2 * u + 1], cr, zi[u]);
          dot2_acc(h[2 * u + 1], l[2 * u + 1], ci, zr[u]);
          l[2 * u + 1] = fmaf(lr, zi[u], fmaf(li, zr[u], l[2 * u + 1]));
        }
      }
      x4[i] = make_float4(h[0] + l[0], h[1] + l[1], h[2] + l[2], h[3] + l[3]);
    }
  } else {
    double cr[K], ci[K];
#pragma unroll
    for (int j = 0; j < K; j++) {
      cr[j] = scale * c[2 * j];
      ci[j] = scale * c[2 * j + 1];
    }
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
      cx<T> a = x[i];
      double re = (double)a.re, im = (double)a.im;
#pragma unroll
      for (int j = 0; j < K; j++) {
        const cx<TZ> z = Z.p[j][i];
        const double zr = (double)z.re, zi = (double)z.im;
        re = fma(cr[j], zr, fma(-ci[j], zi, re));
        im = fma(cr[j], zi, fma(ci[j], zr, im));
      }
      x[i] = mkc<T>((T)re, (T)im);
    }
  }
}

template <typename T, typename TZ>
void blas_lincomb(T* x, const TZ* const* Z, const double* d_c, int k, double scale, size_t n, cudaStream_t s) {
  for (int j0 = 0; j0 < k; j0 += 8) {
    const int kk = (k - j0) < 8 ? (k - j0) : 8;
    VecPtrs<TZ> P;
    for (int j = 0; j < 8; j++) P.p[j] = (const cx<TZ>*)(j < kk ? Z[j0 + j] : Z[j0]);
    const double* c = d_c + 2 * j0;
    const int grid = ew_grid(sizeof(T) == 4 ? n / 2 : n);
    cx<T>* xp = (cx<T>*)x;
    switch (kk) {
      case 1: k_lincomb<T, TZ, 1><<<grid, kBS, 0, s>>>(xp, P, c, scale, n); break;
      case 2: k_lincomb<T, TZ, 2><<<grid, kBS, 0, s>>>(xp, P, c, scale, n); break;
      case 3: k_lincomb<T, TZ, 3><<<grid, kBS, 0, s>>>(xp, P, c, scale, n); break;
      case 4: k_lincomb<T, TZ, 4><<<grid, kBS, 0, s>>>(xp, P, c, scale, n); break;
      case 5: k_lincomb<T, TZ, 5><<<grid, kBS, 0, s>>>(xp, P, c, scale, n); break;
      case 6: k_lincomb<T, TZ, 6><<<grid, kBS, 0, s>>>(xp, P, c, scale, n); break;
      case 7: k_lincomb<T, TZ, 7><<<grid, kBS, 0, s>>>(xp, P, c, scale, n); break;
      default: k_lincomb<T, TZ, 8><<<grid, kBS, 0, s>>>(xp, P, c, scale, n); break;
    }
    MG_LAUNCH();
  }
}

// c = (triangular beta, diagonal gamma)^{-1} alpha, one warp: the column of each
// c_l is taken from all rows above at once, the next column on its way
// meanwhile (one thread row by row took 18 us for 8 and 41 us for 16 unknowns, 10 here,
// mostly trips to L2 and FP64 divisions).  The right-hand sides are kept in
// shared memory up to kBacksub unknowns, beyond in c itself.
constexpr int kBacksub = 256;
__global__ void __launch_bounds__(32) k_backsub(const double* __restrict__ beta, int ld,
                                                const double* __restrict__ alpha, const double* __restrict__ gamma,
                                                int k, double* c) {
  __shared__ double s_acc[2 * kBacksub];
  double* acc = k <= kBacksub ? s_acc : c;
  const int lane = threadIdx.x;
  for (int i = lane; i < k; i += 32) {
    acc[2 * i] = alpha[2 * i];
    acc[2 * i + 1] = alpha[2 * i + 1];
  }
  __syncwarp();
  auto entry = [&](int i, int l) {
    const double* p = beta + 2 * (i + (size_t)ld * l);
    return make_double2(p[0], p[1]);
  };
  double2 next = make_double2(0.0, 0.0);
  double rg_next = 1.0 / gamma[k - 1];
  if (lane < k - 1) next = entry(lane, k - 1);
  for (int l = k - 1; l >= 0; l--) {
    double2 b = next;
    const double cr = acc[2 * l] * rg_next, ci = acc[2 * l + 1] * rg_next;
    if (lane < l - 1) next = entry(lane, l - 1);
    __syncwarp();
    if (lane == 0) {
      c[2 * l] = cr;
      c[2 * l + 1] = ci;
    }
    for (int i = lane; i < l; i += 32) {
      if (i >= 32) b = entry(i, l);
      acc[2 * i] = fma(-b.x, cr, fma(b.y, ci, acc[2 * i]));
      acc[2 * i + 1] = fma(-b.x, ci, fma(-b.y, cr, acc[2 * i + 1]));
    }
    if (l > 0) rg_next = 1.0 / gamma[l - 1];
    __syncwarp();
  }
}

void gcr_backsub(const double* d_beta, int ld, const double* d_alpha, const double* d_gamma, int k, double* d_c,
                 cudaStream_t s) {
  if (k < 1) return;
  k_backsub<<<1, 32, 0, s>>>(d_beta, ld, d_alpha, d_gamma, k, d_c);
  MG_LAUNCH();
}

template <typename T>
__global__ void k_mr_update(cx<T>* e, cx<T>* r, const cx<T>* __restrict__ w, const double* __restrict__ in, size_t n) {
  __shared__ T s_al[2];
  if (threadIdx.x < 2) s_al[threadIdx.x] = (T)(in[1 + threadIdx.x] / (in[0] > 0 ? in[0] : 1.0));
  __syncthreads();
  const T ar = s_al[0], ai = s_al[1];
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    cx<T> rv = r[i], wv = w[i], ev = e[i];
    ev.re = fma(ar, rv.re, fma(-ai, rv.im, ev.re));
    ev.im = fma(ar, rv.im, fma(ai, rv.re, ev.im));
    rv.re = fma(-ar, wv.re, fma(ai, wv.im, rv.re));
    rv.im = fma(-ar, wv.im, fma(-ai, wv.re, rv.im));
    e[i] = ev;
    r[i] = rv;
  }
}
template <typename T>
void blas_mr_update(T* e, T* r, const T* w, const double* d_in, size_t n, cudaStream_t s) {
  k_mr_update<T><<<ew_grid(n), kBS, 0, s>>>((cx<T>*)e, (cx<T>*)r, (const cx<T>*)w, d_in, n);
  MG_LAUNCH();
}

template <typename T>
__global__ void k_normalize(cx<T>* x, const double* __restrict__ nrm2, size_t n) {
  __shared__ T s_f;
  if (threadIdx.x == 0) s_f = (T)(nrm2[0] > 0 ? 1.0 / sqrt(nrm2[0]) : 1.0);
  __syncthreads();
  const T f = s_f;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    cx<T> a = x[i];
    x[i] = mkc<T>(a.re * f, a.im * f);
  }
}
template <typename T>
void blas_normalize(T* x, const double* d_norm2, size_t n, cudaStream_t s) {
  k_normalize<T><<<ew_grid(n), kBS, 0, s>>>((cx<T>*)x, d_norm2, n);
  MG_LAUNCH();
}

// --------------------------------------------------------------------------- instantiations
#define MG_INST(T)                                                                                             \
  template void blas_zero<T>(T*, size_t, cudaStream_t);                                                        \
  template void blas_axpby<T>(double, const T*, double, T*, size_t, cudaStream_t);                             \
  template void blas_norm2<T>(const T*, size_t, double*, Workspace&, cudaStream_t);                            \
  template void blas_cdot<T>(const T*, const T*, size_t, double*, Workspace&, cudaStream_t);                   \
  template void blas_dot2<T>(const T*, const T*, size_t, double*, Workspace&, cudaStream_t);                   \
  template void blas_multidot<T>(const T* const*, int, const T*, size_t, double*, Workspace&, cudaStream_t);   \
  template void blas_orth_update<T>(T*, const T* const*, const double*, int, const T*, size_t, double*,        \
                                    Workspace&, cudaStream_t);                                                 \
  template void blas_r_update<T>(T*, const T*, T*, size_t, const double*, double*, double*, double*, Workspace&, \
                                 cudaStream_t);                                                                \
  template void blas_mr_update<T>(T*, T*, const T*, const double*, size_t, cudaStream_t);                      \
  template void blas_normalize<T>(T*, const double*, size_t, cudaStream_t);
MG_INST(float)
MG_INST(double)
#undef MG_INST
template void blas_convert<float, double>(double*, const float*, size_t, cudaStream_t);
template void blas_convert<double, float>(float*, const double*, size_t, cudaStream_t);
template void blas_convert<float, float>(float*, const float*, size_t, cudaStream_t);
template void blas_convert<double, double>(double*, const double*, size_t, cudaStream_t);
template void blas_lincomb<double, float>(double*, const float* const*, const double*, int, double, size_t,
                                          cudaStream_t);
template void blas_lincomb<double, double>(double*, const double* const*, const double*, int, double, size_t,
                                           cudaStream_t);
template void blas_lincomb<float, float>(float*, const float* const*, const double*, int, double, size_t,
                                         cudaStream_t);

}  // namespace mg
