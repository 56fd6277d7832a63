// Krylov solvers the paper compares multigrid against (section "Results"):
// BiCGStab, CG on the normal equations (CGNR) and, built on BiCGStab, a
// mixed-precision solver by iterative refinement (driven from solver.cu).
// They run on the even-odd reduced operator D_r with the same fine kernels as
// the multigrid solve.  BiCGStab's vector work is four fused passes per
// iteration that form alpha and omega on the device, so the host waits once
// per iteration, for the norms that decide convergence (separate copies,
// linear combinations and three waits with coefficient uploads took 60 us of
// passes and 75 us of gaps in a 280 us iteration of 16^3x32).
#include <algorithm>
#include <complex>

#include "dfloat.cuh"
#include "internal.h"

namespace mg {

namespace {
using cplx = std::complex<double>;

// gamma_5 = diag(1, 1, -1, -1) in spin (chiral basis).  A half vector in the
// internal layout is six chunks of two complex components (component =
// 3 spin + colour), chunk-major over the sites, so spins 2 and 3 are the last
// three chunks: the second half of the vector.
template <typename T>
void gamma5_half(Ctx* c, T* v) {
  T* hi = v + 12 * (size_t)c->Vh;  // 6 Vh complex numbers in
  blas_axpby<T>(0.0, hi, -1.0, hi, 6 * (size_t)c->Vh, c->stream);
}
}  // namespace

// D_r = S A_e^{-1} with S = A_e - H_eo A_o^{-1} H_oe the Schur complement.
// gamma_5-hermiticity of D (H_eo^dag = gamma_5 H_oe gamma_5) and the clover
// blocks being Hermitian and commuting with gamma_5 give S^dag = gamma_5 S
// gamma_5, so D_r^dag = A_e^{-1} gamma_5 S gamma_5 = gamma_5 A_e^{-1} D_r A_e gamma_5.
template <typename T>
void dr_dagger(Ctx* c, FineOps<T>& F, T* out, const T* in, T* tmp) {
  const size_t n = 12 * (size_t)c->Vh;
  blas_convert<T, T>(tmp, in, n, c->stream);
  gamma5_half(c, tmp);
  clover_apply<T>(c->g, out, tmp, c->A<T>(0), c->stream);     // A_e gamma_5 in
  F.Dr(tmp, out);                                               // D_r A_e gamma_5 in
  clover_apply<T>(c->g, out, tmp, c->Ainv<T>(0), c->stream);  // A_e^{-1} D_r A_e gamma_5 in
  gamma5_half(c, out);
}

template <typename T>
Krylov<T>::Krylov(Ctx* c, size_t n) : c_(c), n_(n) {
  for (DBuf* d : {&r_, &rh_, &p_, &v_, &s_, &t_}) {
    d->alloc(sizeof(T) * 2 * n);
    MG_CUDA(cudaMemsetAsync(d->get(), 0, sizeof(T) * 2 * n, c->stream));
  }
  sc_.alloc(sizeof(double) * 16);
}

namespace {
constexpr int kBS = 256;
inline int sum_grid(size_t n) {   // blocks of the fused passes with sums
  const size_t b = (n + kBS - 1) / kBS;
  return (int)(b < 1 ? 1 : (b > (size_t)Workspace::kMaxBlocks ? (size_t)Workspace::kMaxBlocks : b));
}

// device scalars of an iteration (doubles): <rh, v>; <t, t>, <t, s>, ||s||^2;
// <rh, r>, <r, r>; alpha; omega; 1 if <rh, v> broke down
enum { S_RV = 0, S_TT = 2, S_TS = 3, S_SS = 5, S_RHO = 6, S_RR = 8, S_AL = 10, S_OM = 12, S_BROKE = 14, S_COUNT = 15 };

// a complex coefficient and a running sum c z: FP64, or for FP32 vectors the
// coefficient as float pairs and the sum in compensated FP32 (about 48 bits,
// rounded once), as blas_lincomb forms it
template <typename T>
struct Coef;
template <>
struct Coef<double> {
  double re, im;
  __host__ __device__ static Coef of(double r, double i) { return Coef{r, i}; }
};
template <>
struct Coef<float> {
  float rh, rl, ih, il;
  __host__ __device__ static Coef of(double r, double i) {
    const float a = (float)r, b = (float)i;
    return Coef{a, (float)(r - (double)a), b, (float)(i - (double)b)};
  }
};
template <typename T>
struct Sum;
template <>
struct Sum<double> {
  double re, im;
  __device__ explicit Sum(cx<double> z) : re(z.re), im(z.im) {}
  __device__ void add(const Coef<double>& c, cx<double> z) {
    re = fma(c.re, z.re, fma(-c.im, z.im, re));
    im = fma(c.re, z.im, fma(c.im, z.re, im));
  }
  __device__ cx<double> value() const { return mkc(re, im); }
};
template <>
struct Sum<float> {
  float rh, rl, ih, il;
  __device__ explicit Sum(cx<float> z) : rh(z.re), rl(0.f), ih(z.im), il(0.f) {}
  __device__ void add(const Coef<float>& c, cx<float> z) {
    dot2_acc(rh, rl, c.rh, z.re);
    dot2_acc(rh, rl, -c.ih, z.im);
    rl = fmaf(c.rl, z.re, fmaf(-c.il, z.im, rl));
    dot2_acc(ih, il, c.rh, z.im);
    dot2_acc(ih, il, c.ih, z.re);
    il = fmaf(c.rl, z.im, fmaf(c.il, z.re, il));
  }
  __device__ cx<float> value() const { return mkc(rh + rl, ih + il); }
};

// Scalars are products of two vectors and are taken relative to rn^2 (irn = 1 / rn)
// before anything is squared: vectors of any scale that FP64 norms hold.
struct Scaled {
  double re, im;
  __device__ Scaled(double r, double i, double irn) : re((r * irn) * irn), im((i * irn) * irn) {}
  __device__ double abs2() const { return re * re + im * im; }
};

// p = r + beta p - (beta omega) v
template <typename T>
__global__ void __launch_bounds__(kBS) k_bicg_p(cx<T>* __restrict__ p, const cx<T>* __restrict__ r,
                                                const cx<T>* __restrict__ v, Coef<T> beta, Coef<T> mbo, size_t n) {
  for (size_t i = blockIdx.x * (size_t)kBS + threadIdx.x; i < n; i += (size_t)gridDim.x * kBS) {
    Sum<T> s(r[i]);
    s.add(beta, p[i]);
    s.add(mbo, v[i]);
    p[i] = s.value();
  }
}

// s = r - alpha v, alpha = rho / <rh, v> (0 on a breakdown, which the host sees too)
template <typename T>
__global__ void __launch_bounds__(kBS) k_bicg_s(cx<T>* __restrict__ sv, const cx<T>* __restrict__ r,
                                                const cx<T>* __restrict__ v, double rho_re, double rho_im, double irn,
                                                double* sc, size_t n) {
  __shared__ Coef<T> ma;
  if (threadIdx.x == 0) {
    const Scaled rv(sc[S_RV], sc[S_RV + 1], irn), rho(rho_re, rho_im, irn);
    const double a2 = rv.abs2();
    const bool broke = a2 <= 1e-60;   // |<rh, v>| <= 1e-30 rn^2
    double re = 0.0, im = 0.0;
    if (!broke) {
      const double d = 1.0 / a2;
      re = (rho.re * rv.re + rho.im * rv.im) * d;
      im = (rho.im * rv.re - rho.re * rv.im) * d;
    }
    ma = Coef<T>::of(-re, -im);
    if (blockIdx.x == 0) {
      sc[S_AL] = re;
      sc[S_AL + 1] = im;
      sc[S_BROKE] = broke ? 1.0 : 0.0;
    }
  }
  __syncthreads();
  const Coef<T> c = ma;
  for (size_t i = blockIdx.x * (size_t)kBS + threadIdx.x; i < n; i += (size_t)gridDim.x * kBS) {
    Sum<T> s(r[i]);
    s.add(c, v[i]);
    sv[i] = s.value();
  }
}

// {<t, t>, Re <t, s>, Im <t, s>, ||s||^2} -> sc[S_TT ..]
template <typename T>
__global__ void __launch_bounds__(kBS) k_bicg_dots(const cx<T>* __restrict__ t, const cx<T>* __restrict__ sv, size_t n,
                                                   double* partials, unsigned* counter, double* sc) {
  T v[4] = {0, 0, 0, 0};
  for (size_t i = blockIdx.x * (size_t)kBS + threadIdx.x; i < n; i += (size_t)gridDim.x * kBS) {
    const cx<T> a = t[i], b = sv[i];
    v[0] = fma(a.re, a.re, fma(a.im, a.im, v[0]));
    v[1] = fma(a.re, b.re, fma(a.im, b.im, v[1]));
    v[2] = fma(a.re, b.im, fma(-a.im, b.re, v[2]));
    v[3] = fma(b.re, b.re, fma(b.im, b.im, v[3]));
  }
  grid_sum<kBS, 4>(v, partials, counter, sc + S_TT);
}

// omega = <t, s> / <t, t>: x += alpha p + omega s, r = s - omega t; at the half
// step (||s|| <= tol or t = 0) x += alpha p, r = s; on a breakdown nothing.
// Then {<rh, r>, <r, r>} -> sc[S_RHO ..].
template <typename T>
__global__ void __launch_bounds__(kBS) k_bicg_xr(cx<T>* __restrict__ x, cx<T>* __restrict__ r,
                                                 const cx<T>* __restrict__ p, const cx<T>* __restrict__ sv,
                                                 const cx<T>* __restrict__ t, const cx<T>* __restrict__ rh, double irn,
                                                 double tol_abs, size_t n, double* partials, unsigned* counter,
                                                 double* sc) {
  __shared__ Coef<T> s_al, s_om, s_mom;
  __shared__ int s_skip;
  if (threadIdx.x == 0) {
    const bool half = sqrt(sc[S_SS]) <= tol_abs || sc[S_TT] == 0.0;
    double re = 0.0, im = 0.0;
    if (!half) {
      const Scaled ts(sc[S_TS], sc[S_TS + 1], irn);
      const double d = 1.0 / ((sc[S_TT] * irn) * irn);
      re = ts.re * d;
      im = ts.im * d;
    }
    s_skip = sc[S_BROKE] != 0.0;
    s_al = Coef<T>::of(sc[S_AL], sc[S_AL + 1]);
    s_om = Coef<T>::of(re, im);
    s_mom = Coef<T>::of(-re, -im);
    if (blockIdx.x == 0) {
      sc[S_OM] = re;
      sc[S_OM + 1] = im;
    }
  }
  __syncthreads();
  const Coef<T> al = s_al, om = s_om, mom = s_mom;
  T v[3] = {0, 0, 0};
  if (!s_skip)
    for (size_t i = blockIdx.x * (size_t)kBS + threadIdx.x; i < n; i += (size_t)gridDim.x * kBS) {
      const cx<T> si = sv[i];
      Sum<T> a(x[i]);
      a.add(al, p[i]);
      a.add(om, si);
      x[i] = a.value();
      Sum<T> b(si);
      b.add(mom, t[i]);
      const cx<T> ri = b.value(), h = rh[i];
      r[i] = ri;
      v[0] = fma(h.re, ri.re, fma(h.im, ri.im, v[0]));
      v[1] = fma(h.re, ri.im, fma(-h.im, ri.re, v[1]));
      v[2] = fma(ri.re, ri.re, fma(ri.im, ri.im, v[2]));
    }
  grid_sum<kBS, 3>(v, partials, counter, sc + S_RHO);
}
}  // namespace

// BiCGStab (van der Vorst) on A x = b.  Restarts (rh = r, p = v = 0) when
// <rh, r> or <rh, A p> vanishes or omega does, and stops unconverged when the
// breakdown recurs on the restart itself.  Convergence is tested on the
// recursively updated residual at the half step (s) and the full step (r).
template <typename T>
typename Krylov<T>::Result Krylov<T>::bicgstab(const Op& A, T* x, const T* b, bool x0_zero, double tol_abs,
                                               int maxit) {
  Result res;
  cudaStream_t s = c_->stream;
  const size_t n = n_;
  T* r = r_.as<T>();
  T* rh = rh_.as<T>();
  T* p = p_.as<T>();
  T* v = v_.as<T>();
  T* sv = s_.as<T>();
  T* t = t_.as<T>();
  double* d = sc_.as<double>();
  double h[S_COUNT];
  if (x0_zero) {
    blas_zero<T>(x, n, s);
    blas_convert<T, T>(r, b, n, s);
  } else {
    A(r, x);
    blas_axpby<T>(1.0, b, -1.0, r, n, s);  // r = b - A x
  }
  blas_norm2<T>(r, n, d, c_->ws, s);
  double rn = std::sqrt(c_->read_scalar(d));
  res.rnorm = rn;
  if (!std::isfinite(rn)) raise(MG_ERR_NAN, "non-finite residual in BiCGStab");
  if (rn <= tol_abs) {
    res.converged = true;
    return res;
  }
  const int grid = sum_grid(n);
  const unsigned wide = (unsigned)std::min<size_t>(152 * 8, (n + kBS - 1) / kBS);
  double* part = c_->ws.partials.template as<double>();
  unsigned* cnt = c_->ws.counter.template as<unsigned>();
  auto cv = [](T* v) { return reinterpret_cast<cx<T>*>(v); };
  bool fresh = true;
  cplx rho(1.0, 0.0), alpha(1.0, 0.0), omega(1.0, 0.0), rho_new;
  while (res.iterations < maxit) {
    const bool restarted = fresh;
    if (fresh) {
      blas_convert<T, T>(rh, r, n, s);
      blas_convert<T, T>(p, r, n, s);
      rho_new = cplx(rn * rn, 0.0);
    } else {
      const cplx beta = (rho_new / rho) * (alpha / omega), mbo = -beta * omega;
      k_bicg_p<T><<<wide, kBS, 0, s>>>(cv(p), cv(r), cv(v), Coef<T>::of(beta.real(), beta.imag()),
                                       Coef<T>::of(mbo.real(), mbo.imag()), n);
      MG_LAUNCH();
    }
    fresh = false;
    A(v, p);
    blas_cdot<T>(rh, v, n, d + S_RV, c_->ws, s);
    k_bicg_s<T><<<wide, kBS, 0, s>>>(cv(sv), cv(r), cv(v), rho_new.real(), rho_new.imag(), 1.0 / rn, d, n);
    MG_LAUNCH();
    A(t, sv);
    k_bicg_dots<T><<<grid, kBS, 0, s>>>(cv(t), cv(sv), n, part, cnt, d);
    MG_LAUNCH();
    k_bicg_xr<T><<<grid, kBS, 0, s>>>(cv(x), cv(r), cv(p), cv(sv), cv(t), cv(rh), 1.0 / rn, tol_abs, n, part, cnt, d);
    MG_LAUNCH();
    c_->read_scalars(d, h, S_COUNT);
    if (!std::isfinite(h[S_RV]) || !std::isfinite(h[S_RV + 1])) raise(MG_ERR_NAN, "non-finite scalar in BiCGStab");
    if (h[S_BROKE] != 0.0) {
      // breakdown: restart from the current residual, unless this step already
      // was the restart (<r, A r> = 0: no progress possible from here)
      if (restarted) break;
      res.restarts++;
      fresh = true;
      continue;
    }
    res.iterations++;
    const double sn = std::sqrt(h[S_SS]);
    if (!std::isfinite(sn) || !std::isfinite(h[S_TT])) raise(MG_ERR_NAN, "non-finite scalar in BiCGStab");
    if (sn <= tol_abs || h[S_TT] == 0.0) {  // converged at the half step (or A s = 0: s is the exact residual)
      res.rnorm = sn;
      res.converged = sn <= tol_abs;
      if (res.converged) break;
      fresh = true;
      rn = sn;
      res.restarts++;
      continue;
    }
    alpha = cplx(h[S_AL], h[S_AL + 1]);
    omega = cplx(h[S_OM], h[S_OM + 1]);
    rn = std::sqrt(h[S_RR]);
    res.rnorm = rn;
    if (!std::isfinite(rn)) raise(MG_ERR_NAN, "non-finite residual in BiCGStab");
    if (rn <= tol_abs) {
      res.converged = true;
      break;
    }
    rho = rho_new;
    rho_new = cplx(h[S_RHO], h[S_RHO + 1]);
    if (std::abs(omega) == 0.0 || std::abs(rho_new) <= 1e-30 * rn * rn) {
      res.restarts++;
      fresh = true;
    }
  }
  return res;
}

// CG on A^dag A x = A^dag b (CGLS form: the residual r = b - A x is updated
// alongside, and the stopping test is ||r|| <= tol_abs).
template <typename T>
typename Krylov<T>::Result Krylov<T>::cgnr(const Op& A, const Op& Adag, T* x, const T* b, bool x0_zero,
                                           double tol_abs, int maxit) {
  Result res;
  cudaStream_t s = c_->stream;
  const size_t n = n_;
  T* r = r_.as<T>();
  T* z = rh_.as<T>();
  T* p = p_.as<T>();
  T* w = v_.as<T>();
  double* d = sc_.as<double>();
  double h[2];
  if (x0_zero) {
    blas_zero<T>(x, n, s);
    blas_convert<T, T>(r, b, n, s);
  } else {
    A(r, x);
    blas_axpby<T>(1.0, b, -1.0, r, n, s);
  }
  Adag(z, r);
  blas_convert<T, T>(p, z, n, s);
  blas_norm2<T>(r, n, d, c_->ws, s);
  blas_norm2<T>(z, n, d + 1, c_->ws, s);
  c_->read_scalars(d, h, 2);
  double rn = std::sqrt(h[0]), zz = h[1];
  res.rnorm = rn;
  if (!std::isfinite(rn) || !std::isfinite(zz)) raise(MG_ERR_NAN, "non-finite residual in CGNR");
  if (rn <= tol_abs) {
    res.converged = true;
    return res;
  }
  while (res.iterations < maxit && zz > 0.0) {
    A(w, p);
    blas_norm2<T>(w, n, d, c_->ws, s);
    const double ww = c_->read_scalar(d);
    if (!(ww > 0.0) || !std::isfinite(ww)) raise(MG_ERR_NAN, "non-finite or zero <Ap, Ap> in CGNR");
    const double a = zz / ww;
    blas_axpby<T>(a, p, 1.0, x, n, s);
    blas_axpby<T>(-a, w, 1.0, r, n, s);
    Adag(z, r);
    blas_norm2<T>(r, n, d, c_->ws, s);
    blas_norm2<T>(z, n, d + 1, c_->ws, s);
    c_->read_scalars(d, h, 2);
    res.iterations++;
    rn = std::sqrt(h[0]);
    res.rnorm = rn;
    if (!std::isfinite(rn) || !std::isfinite(h[1])) raise(MG_ERR_NAN, "non-finite residual in CGNR");
    if (rn <= tol_abs) {
      res.converged = true;
      break;
    }
    const double beta = h[1] / zz;
    zz = h[1];
    blas_axpby<T>(1.0, z, beta, p, n, s);  // p = z + beta p
  }
  return res;
}

template void dr_dagger<double>(Ctx*, FineOps<double>&, double*, const double*, double*);
template void dr_dagger<float>(Ctx*, FineOps<float>&, float*, const float*, float*);
template class Krylov<double>;
template class Krylov<float>;

}  // namespace mg
