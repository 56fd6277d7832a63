// Double-float arithmetic on the FP32 pipes for reductions that need more
// than single precision: a value is the unevaluated sum h + l of two floats
// (about 48 significant bits), added with error-free transformations (Knuth's
// two-sum, FMA-based two-product).  GB300 runs FP64 at a small fraction of its
// FP32 rate, and these sums sit in every iteration of the persistent
// coarsest-level solvers; the order of every sum is fixed, so results stay
// reproducible bit for bit.
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

namespace mg {

struct df {
  float h, l;
};
__device__ __forceinline__ df df_of(float x) { return df{x, 0.f}; }
__device__ __forceinline__ df df_norm(float s, float e) {   // s + e with |e| small: renormalise
  const float h = s + e;
  return df{h, e - (h - s)};
}
__device__ __forceinline__ df df_add(df a, df b) {
  const float s = a.h + b.h;
  const float bb = s - a.h;
  const float e = (a.h - (s - bb)) + (b.h - bb) + (a.l + b.l);
  return df_norm(s, e);
}
// h + l <- h + l + x, the rounding error of the sum kept in l (not renormalised)
__device__ __forceinline__ void df_acc(float& h, float& l, float x) {
  const float s = __fadd_rn(h, x);
  const float bb = __fsub_rn(s, h);
  l = __fadd_rn(l, __fadd_rn(__fsub_rn(h, __fsub_rn(s, bb)), __fsub_rn(x, bb)));
  h = s;
}
__device__ __forceinline__ df df_neg(df a) { return df{-a.h, -a.l}; }
__device__ __forceinline__ df df_mul(df a, df b) {
  const float p = a.h * b.h;
  const float e = fmaf(a.h, b.h, -p) + (a.h * b.l + a.l * b.h);
  return df_norm(p, e);
}
// a / b (b > 0) by one correction of the float quotient
__device__ __forceinline__ df df_div(df a, df b) {
  const float q1 = a.h / b.h;
  const df r = df_add(a, df_neg(df_mul(df_of(q1), b)));
  return df_norm(q1, r.h / b.h);
}
// sqrt(a), a >= 0, by one Newton correction of sqrtf
__device__ __forceinline__ df df_sqrt(df a) {
  if (!(a.h > 0.f)) return df_of(0.f);
  const float s = sqrtf(a.h);
  const df r = df_add(a, df_neg(df_mul(df_of(s), df_of(s))));
  return df_norm(s, r.h / (2.f * s));
}
// a b added to h + l with the rounding errors of the product and of the sum
// kept in l (Ogita, Rump and Oishi's Dot2, not renormalised)
__device__ __forceinline__ void dot2_acc(float& h, float& l, float a, float b) {
  const float p = __fmul_rn(a, b);
  const float e = fmaf(a, b, -p);
  const float s = __fadd_rn(h, p);
  const float bb = __fsub_rn(s, h);
  const float t = __fadd_rn(__fsub_rn(h, __fsub_rn(s, bb)), __fsub_rn(p, bb));
  l = __fadd_rn(l, __fadd_rn(t, e));
  h = s;
}
// the same for a product of two double-floats (the l l term is below the sum's error)
__device__ __forceinline__ void df_dot_acc(float& h, float& l, df a, df b) {
  const float p = __fmul_rn(a.h, b.h);
  const float e = fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -p)));
  const float s = __fadd_rn(h, p);
  const float bb = __fsub_rn(s, h);
  const float t = __fadd_rn(__fsub_rn(h, __fsub_rn(s, bb)), __fsub_rn(p, bb));
  l = __fadd_rn(l, __fadd_rn(t, e));
  h = s;
}
__device__ __forceinline__ df df_wsum(df v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const df u{__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o)};
    v = df_add(v, u);
  }
  return v;
}

// Sums over the warp of V (2, 4, 8, 16) values per lane by transposition: each
// of the first log2 V levels keeps half of the values and passes the other half
// to its partner, the remaining levels add whole values, so V values cost
// V - 1 + log2(32 / V) additions per lane instead of 5 V.  Lane l ends with the
// warp total of v[(l >> (5 - log2 V)) & (V - 1)], added in a fixed order.
__device__ __forceinline__ float shfl_x(float v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ double shfl_x(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ df shfl_x(df v, int o) { return df{shfl_x(v.h, o), shfl_x(v.l, o)}; }
__device__ __forceinline__ float add_x(float a, float b) { return a + b; }
__device__ __forceinline__ double add_x(double a, double b) { return a + b; }
__device__ __forceinline__ df add_x(df a, df b) { return df_add(a, b); }
template <int V, int LANES = 32, typename S>
__device__ __forceinline__ S warp_transpose_sum(S (&v)[V]) {
  const int lane = threadIdx.x & 31;
  int off = LANES / 2;
#pragma unroll
  for (int half = V / 2; half >= 1; half /= 2, off /= 2) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < half; i++) {
      const S send = up ? v[i] : v[i + half];
      const S keep = up ? v[i + half] : v[i];
      v[i] = add_x(keep, shfl_x(send, off));
    }
  }
  S t = v[0];
#pragma unroll
  for (int o = LANES / 2 / V; o >= 1; o /= 2) t = add_x(t, shfl_x(t, o));
  return t;
}

// Deterministic sum over the grid of NR values per thread into out[0 .. NR):
// transposed warp sums -- double-float for FP32 sums, FP64 for FP64 ones --, the
// warps of a block added in order, block sums in partials[r][block], and the
// last block to finish adds them, one warp per value.  FP64 additions are the
// scarce resource here (1/62 of the FP32 rate): with a whole butterfly per
// value the tree took longer than the memory pass it closes.  A block whose
// float-pair sum leaves FP32's range adds its threads' sums again in FP64.
// THREADS = block size; the counter is 0 at launch and left at 0.
__device__ __forceinline__ double sum_to_double(double v) { return v; }
__device__ __forceinline__ double sum_to_double(df v) { return (double)v.h + (double)v.l; }
__device__ __forceinline__ double sum_of(double v) { return v; }
__device__ __forceinline__ df sum_of(float v) { return df_of(v); }
__device__ __forceinline__ df sum_of(df v) { return v; }
template <int THREADS, int NR, typename T>
__device__ __forceinline__ void grid_sum(const T (&v)[NR], double* partials, unsigned* counter, double* out) {
  using S = decltype(sum_of(T{}));
  constexpr int W = THREADS / 32;
  constexpr int V = NR <= 1 ? 1 : NR <= 2 ? 2 : NR <= 4 ? 4 : NR <= 8 ? 8 : 16;
  static_assert(NR <= 16, "at most 16 values");
  __shared__ __align__(8) S sm[NR][W];
  __shared__ int state;   // 0: not the last block, 1: the last one, 2: out of range
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // the block's sums, written by lanes of the first warp, then its ticket
  auto ticket = [&]() {
    __syncwarp();
    if (lane == 0) {
      __threadfence();   // the block's partials before its ticket
      state = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
  };
  S t[V];
#pragma unroll
  for (int r = 0; r < V; r++) t[r] = r < NR ? sum_of(v[r < NR ? r : 0]) : sum_of(T{});
  S sum;
  if constexpr (V == 1) {
    sum = t[0];
#pragma unroll
    for (int o = 16; o >= 1; o /= 2) sum = add_x(sum, shfl_x(sum, o));
    if (lane == 0) sm[0][wid] = sum;
  } else {
    sum = warp_transpose_sum<V>(t);
    constexpr int per = 32 / V;   // lanes holding one value
    const int r = lane / per;
    if (lane % per == 0 && r < NR) sm[r][wid] = sum;
  }
  __syncthreads();
  if (wid == 0) {
    bool over = false;
    if (lane < NR) {
      S s = sm[lane][0];
#pragma unroll
      for (int w = 1; w < W; w++) s = add_x(s, sm[lane][w]);
      partials[(size_t)lane * gridDim.x + blockIdx.x] = sum_to_double(s);
      if constexpr (!std::is_same<T, double>::value) over = !(fabsf(s.h) <= 3.402823466e38f);
    }
    if (!std::is_same<T, double>::value && __any_sync(0xffffffffu, over)) {
      if (lane == 0) state = 2;
    } else {
      ticket();
    }
  }
  __syncthreads();
  if constexpr (!std::is_same<T, double>::value) {
    if (state == 2) {   // finite sums of threads beyond FP32's range in the block: again in FP64
      double* sd = reinterpret_cast<double*>(&sm[0][0]);
#pragma unroll
      for (int r = 0; r < NR; r++) {
        double d = sum_to_double(sum_of(v[r]));
#pragma unroll
        for (int o = 16; o >= 1; o /= 2) d += __shfl_xor_sync(0xffffffffu, d, o);
        if (lane == 0) sd[r * W + wid] = d;
      }
      __syncthreads();
      if (wid == 0) {
        if (lane < NR) {
          double d = 0.0;
          for (int w = 0; w < W; w++) d += sd[lane * W + w];
          partials[(size_t)lane * gridDim.x + blockIdx.x] = d;
        }
        ticket();
      }
      __syncthreads();
    }
  }
  if (!state) return;
  __threadfence();
  if constexpr (NR <= 4) {   // every thread takes blocks, all values in flight together
    __shared__ double fin[NR][W];
    double s[NR];
#pragma unroll
    for (int r = 0; r < NR; r++) s[r] = 0.0;
#pragma unroll 4
    for (int b = threadIdx.x; b < (int)gridDim.x; b += THREADS)
#pragma unroll
      for (int r = 0; r < NR; r++) s[r] += __ldcg(&partials[(size_t)r * gridDim.x + b]);
#pragma unroll
    for (int r = 0; r < NR; r++) {
#pragma unroll
      for (int o = 16; o >= 1; o /= 2) s[r] += __shfl_xor_sync(0xffffffffu, s[r], o);
      if (lane == 0) fin[r][wid] = s[r];
    }
    __syncthreads();
    if (threadIdx.x < NR) {
      double t = fin[threadIdx.x][0];
#pragma unroll
      for (int w = 1; w < W; w++) t += fin[threadIdx.x][w];
      out[threadIdx.x] = t;
    }
  } else {
    for (int r = wid; r < NR; r += W) {
      double s = 0.0;
#pragma unroll 8
      for (int b = lane; b < (int)gridDim.x; b += 32) s += __ldcg(&partials[(size_t)r * gridDim.x + b]);
#pragma unroll
      for (int o = 16; o >= 1; o /= 2) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) out[r] = s;
    }
  }
  if (threadIdx.x == 0) *counter = 0u;
}

}  // namespace mg
