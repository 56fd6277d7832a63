// The coarsest-level GCR of 1 to 16 systems of one lattice, every link read
// once per application for all of them.
//
// Same method as coarse_gcr.cu (section "Implementation": unpreconditioned
// GCR on the coarsest lattice to a tolerance relative to each right-hand side;
// section "Red-black preconditioning": the reduced even-odd system, or the
// operator itself when an extent is odd), arranged so that an iteration of
// nb systems costs about what its arithmetic costs:
//
//  * Work items are kRows consecutive link rows of one site.  Every block owns
//    a fixed contiguous range of items and, in every element-wise step, the
//    vector elements those rows produce, for all systems: the Gram-Schmidt
//    inner products follow the stencil without a barrier and the Krylov
//    vectors of a block are private to it.
//  * A warp holds kRows x NS complex sums.  Its lanes stride along the rows two
//    complex numbers at a time, the next step's links (16 bytes per row and
//    lane, from L2) in flight while the present ones meet the NS gathered
//    vectors in shared memory: 4 link and NS vector loads per 8 x 4 x NS FMAs,
//    so with NS = 12 the FP32 pipes, not the shared-memory port (67 %), set the
//    time.  One transposed reduction per 32 sums finishes the rows.
//  * Even-odd lattices: phase A applies the folded odd-site links
//    X_o^{-1} Y_d X^{-1}(o + d) (FP32), phase B the even-site links Y_eo in
//    their storage format.  One iteration is
//      phase A | barrier | phase B, inner products | barrier |
//      sums over the blocks, one warp per value | barrier |
//      coefficients, w and r | barrier
//    (with one system every block adds the few sums itself: three barriers).
//    Odd-extent lattices have the one phase w = [Y | X] r.
//  * The norm of the projected w comes from Pythagoras (the w_j are
//    orthonormal), with a second, exact reduction when any system loses more
//    than three digits in it.  The residual before each step is kept as that
//    step's direction and the solution is formed at the end of a restart cycle
//    by back substitution, so an iteration reads the Krylov history twice.
//  * The closing true residual has computed t = A y_e on the odd sites, and
//    x_o = X_o^{-1} (b_o - Y_oe X_e^{-1} y_e) = X_o^{-1} b_o - t.
//
// Measured (16^3x32, 4^4 blocks, Nc = 48, 256 reduced sites, twelve systems,
// 34 iterations): 10.1 ms per launch on the tensor-core kernel, whose site
// inverses and Krylov loops ran on a few warps; 2.33 ms with the next links in
// flight only within an item, the epilogue's reads after the sums and whole
// warps on the inner products; 2.20 ms here, 65 us per iteration of which the
// FMAs of the two stencil phases are 12 and the four barriers 6.  Reductions
// are double-float and added in a fixed order; every wait is bounded in time
// (async_copy.cuh); FLAG_TIMEOUT on expiry.
#include <algorithm>
#include <cstring>

#include "async_copy.cuh"
#include "coarse.h"
#include "coarse_dev.cuh"
#include "dfloat.cuh"

namespace mg {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxRestart = 64;
constexpr int kMaxSys = 16;
constexpr int kRows = 4;
constexpr int kDeep = 6;   // link steps in flight with one system
// reduction slots of a system: <w_j, w> (2 per j), then ||w||^2, Re and Im
// <w, r>, the norm of a right-hand side or true residual, the exact
// ||w''||^2, Re and Im <w'', r>
constexpr int QW = 2 * kMaxRestart;
constexpr int QN = QW + 3;
constexpr int QE = QN + 1;
constexpr int kSlots = QE + 3;

struct GArgs {
  int nc, half, rows_sites, m, maxit, nb, ips, items, chunk;   // rows_sites: sites of the solved system
  float tol_rel[kMaxSys];
  const int* nbr;
  const unsigned char* Y;   // even-site links [e][nc][8][nc], storage format
  const float* Ys;          // their tile scales [e][8]
  const unsigned char* A;   // FP32: folded odd-site links [o - half][nc][8][nc], or [site][nc][9][nc]
  const float2* b[kMaxSys];
  float2* x[kMaxSys];
  float2 *y, *r, *br, *tb, *t;   // [p][n]; tb, t on odd sites
  float2 *W, *R;                 // [k][p][n]
  float2* part;                  // [p * kSlots + slot][block]
  float2* tot;                   // [p * kSlots + slot]
  float2* beta;                  // [p][l][j]
  float2* ag;                    // [p][k]: alpha; then [p][k]: {gamma, -}
  long long* iters[kMaxSys];
  int* flags;
  unsigned* bar;
  int* abort;
};

// gathered vectors of `ns` sites from s0: gv[(site, p)][K] complex, times the
// tile scale; nbd neighbours (8, or 9 with the site itself); in: element
// (storage - base) nc of system p at in + p n.  A warp takes one neighbour of
// one site for all systems (lanes over its nc / 2 <= 32 pairs), 32 neighbours
// to a round: their indices and scales come in one trip to L2, the vectors of
// kPairs neighbours in the next.
template <int NS>
__device__ void gather(const GArgs& a, size_t n, int store0, int s0, int ns, int nbd, int base, const float2* in,
                       const float* scale, float4* gv) {
  constexpr int kPairs = NS <= 4 ? 4 : 2;
  const int hc = a.nc >> 1, K2 = nbd * hc, nt = ns * nbd;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const size_t n2 = n >> 1;
  for (int tb = w; tb < nt; tb += 32 * kWarps) {
    const int tl = min(tb + lane * kWarps, nt - 1), sll = tl / nbd, dl = tl - sll * nbd, stl = store0 + s0 + sll;
    const int froml = dl < 8 ? a.nbr[(size_t)stl * 8 + dl] : stl;
    const float scl = scale && dl < 8 ? scale[(size_t)stl * 8 + dl] : 1.f;
    const int cnt = min(32, (nt - tb + kWarps - 1) / kWarps);
    for (int c = 0; c < cnt; c += kPairs) {
      constexpr int U = NS < 12 ? NS : 12;
#pragma unroll
      for (int p0 = 0; p0 < NS; p0 += U) {
        float4 v[kPairs][U];
#pragma unroll
        for (int x = 0; x < kPairs; x++) {
          const int from = __shfl_sync(0xffffffffu, froml, min(c + x, cnt - 1));
          const float4* src = reinterpret_cast<const float4*>(in) + (size_t)(from - base) * hc + lane;
#pragma unroll
          for (int u = 0; u < U; u++)
            v[x][u] = lane < hc && p0 + u < a.nb ? __ldcg(src + (size_t)(p0 + u) * n2) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int x = 0; x < kPairs; x++) {
          const int cx_ = min(c + x, cnt - 1);   // past the end the last neighbour is written again
          const float sc = __shfl_sync(0xffffffffu, scl, cx_);
          const int t = tb + cx_ * kWarps, sl = t / nbd, d = t - sl * nbd;
          float4* dst = gv + (size_t)sl * NS * K2 + d * hc + lane;
#pragma unroll
          for (int u = 0; u < U; u++)
            if (lane < hc && p0 + u < NS)
              dst[(size_t)(p0 + u) * K2] = make_float4(sc * v[x][u].x, sc * v[x][u].y, sc * v[x][u].z, sc * v[x][u].w);
        }
      }
    }
  }
  __syncthreads();
}

// one stencil phase over the block's items [i0, i1): epi(p, element, value, pre)
// for every row and system, with pre = pre(p, element) read before the item's
// arithmetic (in the epilogue it was three more trips to L2 per item); links of
// site s at links + s nc K entries
template <int ST, int NS, typename Pre, typename Epi>
__device__ void phase(const GArgs& a, size_t n, const unsigned char* links, int i0, int i1, int store0, int nbd,
                      int base, const float2* in, const float* scale, float4* gv, Pre pre, Epi epi) {
  const int nc = a.nc, K2 = nbd * (nc >> 1);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sbeg = i0 / a.ips, send = i1 > i0 ? (i1 - 1) / a.ips + 1 : sbeg;
  for (int s0 = sbeg; s0 < send; s0 += a.chunk) {
    const int ns = min(a.chunk, send - s0);
    gather<NS>(a, n, store0, s0, ns, nbd, base, in, scale, gv);
    const int c0 = max(i0, s0 * a.ips), c1 = min(i1, (s0 + ns) * a.ips);
    using raw_t = typename LinkPair<ST>::raw;
    const unsigned char* row[kRows];
    auto rows_of = [&](int it) {
      const int s = it / a.ips, r0 = (it - s * a.ips) * kRows;
#pragma unroll
      for (int r = 0; r < kRows; r++)   // a row past the end repeats the last one and is dropped
        row[r] = links + ((size_t)s * nc + min(r0 + r, nc - 1)) * (size_t)K2 * sizeof(raw_t);
    };
    auto load = [&](raw_t (&m)[kRows], int q) {
#pragma unroll
      for (int r = 0; r < kRows; r++) m[r] = q < K2 ? LinkPair<ST>::load(row[r], q) : LinkPair<ST>::zero();
    };
    // several systems: the links of the next step are in flight, across items too
    raw_t nx[kRows];
    if (NS > 1 && c0 + w < c1) {
      rows_of(c0 + w);
      load(nx, lane);
    }
    for (int it = c0 + w; it < c1; it += kWarps) {
      const int s = it / a.ips, r0 = (it - s * a.ips) * kRows;
      if (NS == 1) rows_of(it);
      // value f = (r NS + p) 2 + {re, im}: 32 at a time (8 with one system)
      constexpr int V = kRows * NS * 2 < 32 ? kRows * NS * 2 : 32, per = 32 / V, NG = kRows * NS * 2 / V;
      float2 before[NG];
#pragma unroll
      for (int g = 0; g < NG; g++) {
        const int f = g * V + lane / per, r = (f >> 1) / NS, p = (f >> 1) % NS;
        before[g] = lane % (2 * per) == 0 && p < a.nb && r0 + r < nc ? pre(p, (size_t)s * nc + r0 + r) : make_float2(0.f, 0.f);
      }
      float acc[kRows][NS][2];
#pragma unroll
      for (int r = 0; r < kRows; r++)
#pragma unroll
        for (int p = 0; p < NS; p++) acc[r][p][0] = acc[r][p][1] = 0.f;
      const float4* v = gv + (size_t)(s - s0) * NS * K2;
      auto step = [&](const raw_t (&raw)[kRows], int q) {
        float4 l[kRows];
#pragma unroll
        for (int r = 0; r < kRows; r++) l[r] = LinkPair<ST>::decode(raw[r]);
#pragma unroll
        for (int p = 0; p < NS; p++) {
          const float4 x = v[p * K2 + q];
#pragma unroll
          for (int r = 0; r < kRows; r++) {
            acc[r][p][0] = fmaf(l[r].x, x.x, acc[r][p][0]);
            acc[r][p][1] = fmaf(l[r].x, x.y, acc[r][p][1]);
            acc[r][p][0] = fmaf(-l[r].y, x.y, acc[r][p][0]);
            acc[r][p][1] = fmaf(l[r].y, x.x, acc[r][p][1]);
            acc[r][p][0] = fmaf(l[r].z, x.z, acc[r][p][0]);
            acc[r][p][1] = fmaf(l[r].z, x.w, acc[r][p][1]);
            acc[r][p][0] = fmaf(-l[r].w, x.w, acc[r][p][0]);
            acc[r][p][1] = fmaf(l[r].w, x.z, acc[r][p][1]);
          }
        }
      };
      if constexpr (NS == 1) {
        // one system: bound by the links' way from L2, so a lane keeps up to
        // kDeep steps of all rows in flight (98 KB per SM)
        for (int q0 = lane; q0 < K2; q0 += 32 * kDeep) {
          raw_t raw[kDeep][kRows];
#pragma unroll
          for (int u = 0; u < kDeep; u++) load(raw[u], q0 + 32 * u);
#pragma unroll
          for (int u = 0; u < kDeep; u++)
            if (q0 + 32 * u < K2) step(raw[u], q0 + 32 * u);
        }
      } else {
        raw_t cur[kRows];
        for (int q0 = 0; q0 < K2; q0 += 32) {
#pragma unroll
          for (int r = 0; r < kRows; r++) cur[r] = nx[r];
          if (q0 + 32 < K2) {
            load(nx, q0 + 32 + lane);
          } else if (it + kWarps < c1) {
            rows_of(it + kWarps);
            load(nx, lane);
          }
          if (q0 + lane < K2) step(cur, q0 + lane);
        }
      }
#pragma unroll
      for (int g = 0; g < NG; g++) {
        float val[V];
#pragma unroll
        for (int i = 0; i < V; i++) {
          const int f = g * V + i;
          val[i] = acc[(f >> 1) / NS][(f >> 1) % NS][f & 1];
        }
        const float re = warp_transpose_sum<V>(val);
        const float im = __shfl_down_sync(0xffffffffu, re, per);
        const int f = g * V + lane / per;
        const int r = (f >> 1) / NS, p = (f >> 1) % NS;
        if (lane % (2 * per) == 0 && p < a.nb && r0 + r < nc) epi(p, (size_t)s * nc + r0 + r, make_float2(re, im), before[g]);
      }
    }
    __syncthreads();
  }
}

// first element (of a system's vector) of item i
__device__ __forceinline__ size_t item_elem(const GArgs& a, int i) {
  return (size_t)(i / a.ips) * a.nc + (size_t)(i % a.ips) * kRows;
}

// sums of the slots [q0, q0 + nq) and [q1, q1 + nq1) of the systems in `mask`
// over the blocks into dst (shared, [nb][kSlots], at the same slots), identical
// in every block.
// Several systems: one warp of the grid per value, a barrier, and every block
// reads the sums; one system: every block adds the partials itself.
template <int NS>
__device__ bool grid_totals(const GArgs& a, unsigned mask, int q0, int nq, int q1, int nq1, df* dst,
                            unsigned& target) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, G = gridDim.x;
  const int nqt = nq + nq1;
  auto slot_of = [&](int q) { return q < nq ? q0 + q : q1 + (q - nq); };
  auto one = [&](int slot) {
    const float2* p = a.part + (size_t)slot * G;
    df s = df_of(0.f);
    for (int g0 = 0; g0 < G; g0 += 256) {
      float2 t[8];
#pragma unroll
      for (int i = 0; i < 8; i++) {
        const int g = g0 + 32 * i + lane;
        t[i] = g < G ? __ldcg(p + g) : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int i = 0; i < 8; i++) s = df_add(s, df{t[i].x, t[i].y});
    }
    return df_wsum(s);
  };
  if (NS == 1) {
    for (int q = wid; q < nqt; q += kWarps) {
      const df s = one(slot_of(q));
      if (lane == 0) dst[slot_of(q)] = s;
    }
    __syncthreads();
    return true;
  }
  for (int v = blockIdx.x * kWarps + wid; v < a.nb * nqt; v += G * kWarps) {
    const int p = v / nqt, slot = p * kSlots + slot_of(v - p * nqt);
    if (!((mask >> p) & 1u)) continue;
    const df s = one(slot);
    if (lane == 0) a.tot[slot] = make_float2(s.h, s.l);
  }
  if (!grid_barrier(a.bar, a.abort, target)) return false;
  for (int v = threadIdx.x; v < a.nb * nqt; v += kThreads) {
    const int p = v / nqt, slot = p * kSlots + slot_of(v - p * nqt);
    if (!((mask >> p) & 1u)) continue;
    const float2 x = __ldcg(a.tot + slot);
    dst[slot] = df{x.x, x.y};
  }
  __syncthreads();
  return true;
}

template <int ST, int NS, bool EO>
__global__ void __launch_bounds__(kThreads, 1) k_coarse_gcr_group(GArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ float s_ig[kMaxSys], s_ar[kMaxSys], s_ai[kMaxSys], s_tol2[kMaxSys];
  __shared__ df s_rn[kMaxSys], s_g2[kMaxSys];
  __shared__ int s_its[kMaxSys], s_kp[kMaxSys], s_exact;
  __shared__ unsigned s_act, s_run;
  float4* gv = reinterpret_cast<float4*>(smem);
  const int nc = a.nc, m = a.m, nb = a.nb, G = gridDim.x, bid = blockIdx.x;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nbd = EO ? 8 : 9;
  df* tot = reinterpret_cast<df*>(gv + (size_t)a.chunk * NS * nbd * (nc >> 1));   // [nb][kSlots]
  float2* sbeta = reinterpret_cast<float2*>(tot + (size_t)nb * kSlots);           // [nb][kMaxRestart]
  const size_t n = (size_t)a.rows_sites * nc;
  const int i0 = (int)((long long)bid * a.items / G), i1 = (int)((long long)(bid + 1) * a.items / G);
  const size_t E0 = item_elem(a, i0), E1 = i1 == a.items ? n : item_elem(a, i1);
  const int E = (int)(E1 - E0), E2 = E >> 1;   // both ends are even: pairs of elements, 16-byte accesses
  unsigned target = 0;
  bool ok = true;
  auto Wk = [&](int k, int p) { return a.W + ((size_t)k * nb + p) * n + E0; };
  auto Rk = [&](int k, int p) { return a.R + ((size_t)k * nb + p) * n + E0; };
  auto partial = [&](int p, int q, df s) { a.part[((size_t)p * kSlots + q) * G + bid] = make_float2(s.h, s.l); };
  // w = D v for all systems: t on the odd sites, a barrier, out(p, element, Y_eo t); or out(p, element, D_hat v)
  auto none = [](int, size_t) { return make_float2(0.f, 0.f); };
  auto apply = [&](const float2* in, auto pre, auto out) -> bool {
    if (EO) {
      phase<kStF32, NS>(a, n, a.A, i0, i1, a.half, 8, 0, in, nullptr, gv, none,
                        [&](int p, size_t e, float2 u, float2) { a.t[(size_t)p * n + e] = u; });
      if (!grid_barrier(a.bar, a.abort, target)) return false;
      phase<ST, NS>(a, n, a.Y, i0, i1, 0, 8, a.half, a.t, a.Ys, gv, pre, out);
    } else {
      phase<kStF32, NS>(a, n, a.A, i0, i1, 0, 9, 0, in, nullptr, gv, pre, out);
    }
    return true;
  };
  // the block's sum of per-lane values of one warp, into slot q of system p
  auto warp_norm = [&](const float2* v, int p, int q) {   // ||v||^2 over the owned elements of system p
    float s = 0.f;
    for (int e = lane; e < E; e += 32) {
      const float2 x = __ldcg(v + e);
      s = fmaf(x.x, x.x, fmaf(x.y, x.y, s));
    }
    const df t = df_wsum(df_of(s));
    if (lane == 0) partial(p, q, t);
  };

  if (threadIdx.x < kMaxSys) {
    s_its[threadIdx.x] = 0;
    s_rn[threadIdx.x] = df_of(0.f);
  }
  // ||b_p||^2 (any partition of the full right-hand sides)
  for (int p = wid; p < nb; p += kWarps) {
    const size_t nf = EO ? 2 * n : n, cf = (nf + G - 1) / G;
    const size_t f0 = (size_t)bid * cf, f1 = f0 + cf < nf ? f0 + cf : nf;
    float s = 0.f;
    for (size_t e = f0 + lane; e < f1; e += 32) {
      const float2 q = a.b[p][e];
      s = fmaf(q.x, q.x, fmaf(q.y, q.y, s));
    }
    const df t = df_wsum(df_of(s));
    if (lane == 0) partial(p, QN, t);
  }
  // r = b_r = b_e - Y_eo X_o^{-1} b_o (or b), y = 0 on the owned elements
  if (EO)
    phase<ST, NS>(a, n, a.Y, i0, i1, 0, 8, a.half, a.tb, a.Ys, gv, [&](int p, size_t e) { return a.b[p][e]; },
                  [&](int p, size_t e, float2 u, float2 bb) {
      a.br[(size_t)p * n + e] = make_float2(bb.x - u.x, bb.y - u.y);
    });
  for (int q = threadIdx.x; q < nb * E; q += kThreads) {
    const int p = q / E;
    const size_t i = (size_t)p * n + E0 + (q - p * E);
    const float2 bb = EO ? a.br[i] : a.b[p][E0 + (q - p * E)];
    if (!EO) a.br[i] = bb;
    a.r[i] = bb;
    a.y[i] = make_float2(0.f, 0.f);
  }
  __syncthreads();
  for (int p = wid; p < nb; p += kWarps) warp_norm(a.r + (size_t)p * n + E0, p, QE);
  ok = grid_barrier(a.bar, a.abort, target);
  const unsigned all = (1u << nb) - 1u;
  if (ok) ok = grid_totals<NS>(a, all, QN, 2, 0, 0, tot, target);   // ||b||^2 and ||b_r||^2
  if (ok && threadIdx.x == 0) {
    unsigned act = 0u;
    for (int p = 0; p < nb; p++) {
      const df b2 = tot[p * kSlots + QN];
      s_tol2[p] = a.tol_rel[p] * a.tol_rel[p] * (b2.h + b2.l);
      s_rn[p] = tot[p * kSlots + QE];
      if (b2.h > 0.f) act |= 1u << p;
      if (!(s_rn[p].h == s_rn[p].h)) {   // NaN or infinity in b: nothing to iterate on
        act &= ~(1u << p);
        atomicExch(&a.flags[FLAG_NAN], 1);
      }
    }
    s_act = act;
  }
  __syncthreads();
  bool have_t = false;
  int its = 0;
  while (ok && s_act && its < a.maxit) {
    int k = 0;
    if (threadIdx.x == 0) s_run = s_act;
    if (threadIdx.x < kMaxSys) s_kp[threadIdx.x] = 0;
    __syncthreads();
    while (k < m && its < a.maxit && s_run) {
      const unsigned run = s_run;
      // w = D r into the history slot, on the owned elements
      if (!(ok = apply(a.r, [&](int p, size_t e) { return EO ? a.r[(size_t)p * n + e] : make_float2(0.f, 0.f); },
                       [&](int p, size_t e, float2 u, float2 rr) {
              if (EO) u = make_float2(rr.x - u.x, rr.y - u.y);
              a.W[((size_t)k * nb + p) * n + e] = u;
            })))
        break;
      // <w_j, w> (a half-warp takes four j of one system, two elements per load: 16
      // lanes leave fewer of them idle on a short slice and half the sums to
      // reduce per lane), ||w||^2 and <w, r>
      const int groups = max(1, (k + 7) >> 3), l16 = lane & 15;
      for (int task = wid; task < nb * groups; task += kWarps) {
        const int p = task % nb, gi = task / nb;
        if (!((run >> p) & 1u)) continue;
        const float4* wk = reinterpret_cast<const float4*>(Wk(k, p));
        const float4* rp = reinterpret_cast<const float4*>(a.r + (size_t)p * n + E0);
        const int j0 = 8 * gi + 4 * (lane >> 4);
        float re[4], im[4], s0 = 0.f, s1 = 0.f, s2 = 0.f;
#pragma unroll
        for (int u = 0; u < 4; u++) re[u] = im[u] = 0.f;
#pragma unroll 3
        for (int e = l16; e < E2; e += 16) {
          float4 q[4];
#pragma unroll
          for (int u = 0; u < 4; u++)
            q[u] = j0 + u < k ? __ldcg(reinterpret_cast<const float4*>(Wk(j0 + u, p)) + e) : make_float4(0.f, 0.f, 0.f, 0.f);
          const float4 x = __ldcg(wk + e);
          if (gi == 0 && lane < 16) {
            const float4 rr = __ldcg(rp + e);
            s0 = fmaf(x.x, x.x, fmaf(x.y, x.y, fmaf(x.z, x.z, fmaf(x.w, x.w, s0))));
            s1 = fmaf(x.x, rr.x, fmaf(x.y, rr.y, fmaf(x.z, rr.z, fmaf(x.w, rr.w, s1))));
            s2 = fmaf(x.x, rr.y, fmaf(-x.y, rr.x, fmaf(x.z, rr.w, fmaf(-x.w, rr.z, s2))));
          }
#pragma unroll
          for (int u = 0; u < 4; u++) {
            re[u] = fmaf(q[u].x, x.x, fmaf(q[u].y, x.y, fmaf(q[u].z, x.z, fmaf(q[u].w, x.w, re[u]))));
            im[u] = fmaf(q[u].x, x.y, fmaf(-q[u].y, x.x, fmaf(q[u].z, x.w, fmaf(-q[u].w, x.z, im[u]))));
          }
        }
        if (k > 0) {
          df v[8];
#pragma unroll
          for (int u = 0; u < 4; u++) {
            v[2 * u] = df_of(re[u]);
            v[2 * u + 1] = df_of(im[u]);
          }
          const df t = warp_transpose_sum<8, 16>(v);   // lane l of a half: value l >> 1
          const int q = 2 * j0 + (l16 >> 1);
          if ((l16 & 1) == 0 && q < 2 * k) partial(p, q, t);
        }
        if (gi == 0) {
          df v[4] = {df_of(s0), df_of(s1), df_of(s2), df_of(0.f)};
          const df t = warp_transpose_sum<4, 16>(v);   // lane l of a half: value l >> 2
          if ((lane & 3) == 0 && (lane >> 2) < 3) partial(p, QW + (lane >> 2), t);
        }
      }
      if (!(ok = grid_barrier(a.bar, a.abort, target))) break;
      if (!(ok = grid_totals<NS>(a, run, 0, 2 * k, QW, 3, tot, target))) break;
      if (threadIdx.x == 0) s_exact = 0;
      __syncthreads();
      for (int p = wid; p < nb; p += kWarps) {
        if (!((run >> p) & 1u)) continue;
        const df* tp = tot + (size_t)p * kSlots;
        df bb = df_of(0.f);
        for (int j = lane; j < k; j += 32) {
          bb = df_add(bb, df_mul(tp[2 * j], tp[2 * j]));
          bb = df_add(bb, df_mul(tp[2 * j + 1], tp[2 * j + 1]));
          const float2 f = make_float2(tp[2 * j].h + tp[2 * j].l, tp[2 * j + 1].h + tp[2 * j + 1].l);
          sbeta[p * kMaxRestart + j] = f;
          if (bid == p % G) a.beta[((size_t)p * kMaxRestart + k) * kMaxRestart + j] = f;
        }
        bb = df_wsum(bb);
        if (lane == 0) {
          const df g2 = df_add(tp[QW], df_neg(bb));
          s_g2[p] = g2;
          if (!(g2.h > 1e-3f * tp[QW].h)) atomicExch(&s_exact, 1);   // more than three digits lost
        }
      }
      __syncthreads();
      const bool exact = s_exact != 0;   // uniform: from the same totals in every block
      auto finish = [&](int p, int e, float4 x) {   // w_k = w'' / gamma, the direction r, r -= alpha w_k
        float4* rp = reinterpret_cast<float4*>(a.r + (size_t)p * n + E0) + e;
        const float ig = s_ig[p], ar = s_ar[p], ai = s_ai[p];
        x.x *= ig;
        x.y *= ig;
        x.z *= ig;
        x.w *= ig;
        reinterpret_cast<float4*>(Wk(k, p))[e] = x;
        float4 rr = *rp;
        reinterpret_cast<float4*>(Rk(k, p))[e] = rr;
        rr.x -= ar * x.x - ai * x.y;
        rr.y -= ar * x.y + ai * x.x;
        rr.z -= ar * x.z - ai * x.w;
        rr.w -= ar * x.w + ai * x.z;
        *rp = rr;
      };
      auto coefficients = [&]() {
        if (threadIdx.x < nb && ((run >> threadIdx.x) & 1u)) {
          const int p = threadIdx.x;
          const df* d = tot + (size_t)p * kSlots + (exact ? QE + 1 : QW + 1);
          const df g2 = exact ? tot[(size_t)p * kSlots + QE] : s_g2[p];
          const df g = df_sqrt(g2);
          const bool gz = !(g.h > 0.f);
          const df ar = gz ? d[0] : df_div(d[0], g), ai = gz ? d[1] : df_div(d[1], g);
          s_ig[p] = gz ? 1.f : 1.f / g.h;
          s_ar[p] = ar.h + ar.l;
          s_ai[p] = ai.h + ai.l;
          if (!(g2.h == g2.h)) {   // NaN in w: the system ends with this step
            s_rn[p] = g2;
          } else if (!gz) {   // ||r - alpha w_k||^2 = ||r||^2 - |alpha|^2
            const df rn = df_add(s_rn[p], df_neg(df_add(df_mul(ar, ar), df_mul(ai, ai))));
            s_rn[p] = rn.h > 0.f ? rn : df_of(rn.h == rn.h ? 0.f : rn.h);
          }
          if (bid == p % G) {
            a.ag[(size_t)p * kMaxRestart + k] = make_float2(s_ar[p], s_ai[p]);
            a.ag[(size_t)(kMaxSys + p) * kMaxRestart + k] = make_float2(gz ? 1.f : g.h, 0.f);
          }
        }
        __syncthreads();
      };
      if (!exact) coefficients();
      for (int q = threadIdx.x; q < nb * E2; q += kThreads) {
        const int p = q / E2, e = q - p * E2;
        if (!((run >> p) & 1u)) continue;
        float4 x = __ldcg(reinterpret_cast<const float4*>(Wk(k, p)) + e);
        float4 s0 = make_float4(0.f, 0.f, 0.f, 0.f), s1 = s0;
        const float2* bp = sbeta + p * kMaxRestart;
        const float4* hist = reinterpret_cast<const float4*>(Wk(0, p)) + e;
        const size_t step = (size_t)nb * n >> 1;
        auto add = [](float4& s, float2 b, float4 h) {
          s.x = fmaf(b.x, h.x, fmaf(-b.y, h.y, s.x));
          s.y = fmaf(b.x, h.y, fmaf(b.y, h.x, s.y));
          s.z = fmaf(b.x, h.z, fmaf(-b.y, h.w, s.z));
          s.w = fmaf(b.x, h.w, fmaf(b.y, h.z, s.w));
        };
        int j = 0;
        constexpr int U = 16;   // history loads in flight
        for (; j + U <= k; j += U) {
          float4 h[U];
#pragma unroll
          for (int u = 0; u < U; u++) h[u] = __ldcg(hist + (size_t)(j + u) * step);
#pragma unroll
          for (int u = 0; u < U; u += 2) {
            add(s0, bp[j + u], h[u]);
            add(s1, bp[j + u + 1], h[u + 1]);
          }
        }
        if (j < k) {
          float4 h[U];
#pragma unroll
          for (int u = 0; u < U; u++) h[u] = j + u < k ? __ldcg(hist + (size_t)(j + u) * step) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int u = 0; u < U; u++)
            if (j + u < k) add(u & 1 ? s1 : s0, bp[j + u], h[u]);
        }
        x.x -= s0.x + s1.x;
        x.y -= s0.y + s1.y;
        x.z -= s0.z + s1.z;
        x.w -= s0.w + s1.w;
        if (exact)
          reinterpret_cast<float4*>(Wk(k, p))[e] = x;
        else
          finish(p, e, x);
      }
      if (exact) {
        __syncthreads();
        for (int p = wid; p < nb; p += kWarps) {
          if (!((run >> p) & 1u)) continue;
          const float2 *wk = Wk(k, p), *rp = a.r + (size_t)p * n + E0;
          float s0 = 0.f, s1 = 0.f, s2 = 0.f;
          for (int e = lane; e < E; e += 32) {
            const float2 x = __ldcg(wk + e), rr = __ldcg(rp + e);
            s0 = fmaf(x.x, x.x, fmaf(x.y, x.y, s0));
            s1 = fmaf(x.x, rr.x, fmaf(x.y, rr.y, s1));
            s2 = fmaf(x.x, rr.y, fmaf(-x.y, rr.x, s2));
          }
          df v[4] = {df_of(s0), df_of(s1), df_of(s2), df_of(0.f)};
          const df t = warp_transpose_sum<4>(v);
          if ((lane & 7) == 0 && (lane >> 3) < 3) partial(p, QE + (lane >> 3), t);
        }
        if (!(ok = grid_barrier(a.bar, a.abort, target))) break;
        if (!(ok = grid_totals<NS>(a, run, QE, 3, 0, 0, tot, target))) break;
        coefficients();
        for (int q = threadIdx.x; q < nb * E2; q += kThreads) {
          const int p = q / E2, e = q - p * E2;
          if ((run >> p) & 1u) finish(p, e, __ldcg(reinterpret_cast<const float4*>(Wk(k, p)) + e));
        }
      }
      // r complete on every block before the next product reads it
      if (!(ok = grid_barrier(a.bar, a.abort, target))) break;
      k++;
      its++;
      if (threadIdx.x < nb && ((run >> threadIdx.x) & 1u)) {
        const int p = threadIdx.x;
        s_its[p]++;
        s_kp[p] = k;
        const float rn2 = s_rn[p].h;
        if (!(rn2 == rn2)) atomicExch(&a.flags[FLAG_NAN], 1);
        if (!(rn2 == rn2)) atomicAnd(&s_act, ~(1u << p));
        if (!(rn2 > s_tol2[p])) atomicAnd(&s_run, ~(1u << p));
      }
      __syncthreads();
    }
    if (!ok) break;
    // c_j = (alpha_j - sum_{l > j} beta_{j, l} c_l) / gamma_j, a warp per system; then y += sum_j c_j r_j
    for (int p = wid; p < nb; p += kWarps) {
      const int kp = s_kp[p];
      float2* c = sbeta + p * kMaxRestart;
      const float2* be = a.beta + (size_t)p * kMaxRestart * kMaxRestart;
      for (int j = kp - 1; j >= 0; j--) {
        float re = 0.f, im = 0.f;
        for (int l = j + 1 + lane; l < kp; l += 32) {
          const float2 b = __ldcg(be + (size_t)l * kMaxRestart + j), cl = c[l];
          re = fmaf(b.x, cl.x, fmaf(-b.y, cl.y, re));
          im = fmaf(b.x, cl.y, fmaf(b.y, cl.x, im));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          re += __shfl_xor_sync(0xffffffffu, re, o);
          im += __shfl_xor_sync(0xffffffffu, im, o);
        }
        if (lane == 0) {
          const float2 al = __ldcg(a.ag + (size_t)p * kMaxRestart + j);
          const float ig = 1.f / __ldcg(a.ag + (size_t)(kMaxSys + p) * kMaxRestart + j).x;
          c[j] = make_float2((al.x - re) * ig, (al.y - im) * ig);
        }
        __syncwarp();
      }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < nb * E; q += kThreads) {
      const int p = q / E, e = q - p * E, kp = s_kp[p];
      const float2* c = sbeta + p * kMaxRestart;
      const size_t i = (size_t)p * n + E0 + e;
      float2 yy = a.y[i];
      constexpr int U = 16;
      for (int j0 = 0; j0 < kp; j0 += U) {
        float2 z[U];
#pragma unroll
        for (int u = 0; u < U; u++) z[u] = j0 + u < kp ? __ldcg(Rk(j0 + u, p) + e) : make_float2(0.f, 0.f);
#pragma unroll
        for (int u = 0; u < U; u++) {
          const float2 cj = j0 + u < kp ? c[j0 + u] : make_float2(0.f, 0.f);
          yy.x = fmaf(cj.x, z[u].x, fmaf(-cj.y, z[u].y, yy.x));
          yy.y = fmaf(cj.x, z[u].y, fmaf(cj.y, z[u].x, yy.y));
        }
      }
      a.y[i] = yy;
    }
    if (!(ok = grid_barrier(a.bar, a.abort, target))) break;
    // the true residual restarts r and its norm
    if (!(ok = apply(a.y, none, [&](int p, size_t e, float2 u, float2) {
            const size_t i = (size_t)p * n + e;
            if (EO) {
              const float2 yy = a.y[i];
              u = make_float2(yy.x - u.x, yy.y - u.y);
            }
            const float2 bb = a.br[i];
            a.r[i] = make_float2(bb.x - u.x, bb.y - u.y);
          })))
      break;
    have_t = true;
    for (int p = wid; p < nb; p += kWarps) warp_norm(a.r + (size_t)p * n + E0, p, QN);
    if (!(ok = grid_barrier(a.bar, a.abort, target))) break;
    const unsigned act = s_act;
    if (!(ok = grid_totals<NS>(a, act, QN, 1, 0, 0, tot, target))) break;
    if (threadIdx.x < nb && ((act >> threadIdx.x) & 1u)) {
      const int p = threadIdx.x;
      s_rn[p] = tot[(size_t)p * kSlots + QN];
      if (!(s_rn[p].h == s_rn[p].h)) atomicExch(&a.flags[FLAG_NAN], 1);
      if (!(s_rn[p].h > s_tol2[p])) atomicAnd(&s_act, ~(1u << p));
    }
    __syncthreads();
  }
  if (ok) {   // x on the odd sites (x_e = X_e^{-1} y follows in its own launch), or x = y
    for (int q = threadIdx.x; q < nb * E; q += kThreads) {
      const int p = q / E;
      const size_t e = E0 + (q - p * E), i = (size_t)p * n + e;
      if (EO) {
        float2 o = a.tb[i];
        if (have_t) {
          const float2 u = a.t[i];
          o.x -= u.x;
          o.y -= u.y;
        }
        a.x[p][n + e] = o;
      } else {
        a.x[p][e] = a.y[i];
      }
    }
  }
  if (!ok && threadIdx.x == 0) {
    atomicExch(&a.flags[FLAG_TIMEOUT], 1);
    atomicExch(a.abort, 1);
  }
  if (bid == 0 && threadIdx.x < nb)
    atomicAdd(reinterpret_cast<unsigned long long*>(a.iters[threadIdx.x]), (unsigned long long)s_its[threadIdx.x]);
}

// out_p = M(s) in_p for the site blocks M of sites [s0, s1): in_p at element
// (s - in0) nc, out_p at (s - out0) nc.  One CTA per site, its matrix read
// once for every system.
struct SysPtrs {
  const float2* in[kMaxSys];
  float2* out[kMaxSys];
};
__global__ void __launch_bounds__(kThreads) k_site_mul_systems(int nc, int nb, int s0, int in0, int out0,
                                                               const float2* __restrict__ M, SysPtrs v) {
  extern __shared__ __align__(16) float2 sv[];   // [nb][nc]
  const int s = s0 + blockIdx.x;
  for (int t = threadIdx.x; t < nb * nc; t += kThreads)
    sv[t] = v.in[t / nc][(size_t)(s - in0) * nc + t % nc];
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  constexpr int RB = 2, PB = 4;
  for (int i0 = w * RB; i0 < nc; i0 += kWarps * RB)
    for (int p0 = 0; p0 < nb; p0 += PB) {
      const int np = min(PB, nb - p0);
      float2 res[RB][PB];
      warp_gemv_multi<kStF32, RB, PB>(M + (size_t)s * nc * nc, i0, nc, nc, sv + (size_t)p0 * nc, nc, np, lane, res);
      if (lane == 0)
#pragma unroll
        for (int r = 0; r < RB; r++)
          if (i0 + r < nc)
#pragma unroll
            for (int p = 0; p < PB; p++)
              if (p < np) v.out[p0 + p][(size_t)(s - out0) * nc + i0 + r] = res[r][p];
    }
}

int ns_for(int nb) { return nb <= 1 ? 1 : (nb + 3) / 4 * 4; }

struct Plan {
  int grid, items, ips, chunk;
  size_t smem;
};

Plan make_plan(const LevelGeom& G, int nc, int nb) {
  Plan p;
  int dev = 0, optin = 0, sms = 0;
  MG_CUDA(cudaGetDevice(&dev));
  MG_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  MG_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int NS = ns_for(nb);
  p.ips = (nc + kRows - 1) / kRows;
  p.items = (G.eo ? G.half : G.nsites) * p.ips;
  p.grid = std::min(sms, p.items);
  if (NS > 1) {
    // bound by arithmetic: the fewest blocks with the same largest number of
    // items per warp (a barrier costs less with fewer blocks)
    auto rounds = [&](int g) { return ((p.items + g - 1) / g + kWarps - 1) / kWarps; };
    const int most = rounds(p.grid);
    while (p.grid > 1 && rounds(p.grid - 1) == most) p.grid--;
  }
  const size_t fixed = sizeof(df) * (size_t)nb * kSlots + sizeof(float2) * (size_t)nb * kMaxRestart;
  const size_t site = sizeof(float2) * (size_t)NS * (G.eo ? 8 : 9) * nc;
  const size_t budget = (size_t)optin - 2048;   // static shared memory and slack
  const int touched = (int)((p.items + p.grid - 1) / p.grid + p.ips - 2) / p.ips + 1;   // sites a block's items span
  p.chunk = fixed + site <= budget ? (int)std::min<size_t>((budget - fixed) / site, (size_t)std::max(1, touched)) : 0;
  p.smem = fixed + site * (size_t)std::max(1, p.chunk);
  return p;
}

template <int ST, bool EO>
const void* kernel_ns(int NS) {
  switch (NS) {
    case 1: return (const void*)k_coarse_gcr_group<ST, 1, EO>;
    case 4: return (const void*)k_coarse_gcr_group<ST, 4, EO>;
    case 8: return (const void*)k_coarse_gcr_group<ST, 8, EO>;
    case 12: return (const void*)k_coarse_gcr_group<ST, 12, EO>;
    default: return (const void*)k_coarse_gcr_group<ST, 16, EO>;
  }
}
const void* kernel_for(bool eo, int store, int NS) {
  if (!eo) return kernel_ns<kStF32, false>(NS);   // the concatenated links are FP32 in every storage format
  return store == STORE_F16 ? kernel_ns<kStF16, true>(NS)
         : store == STORE_BF16 ? kernel_ns<kStBF16, true>(NS) : kernel_ns<kStF32, true>(NS);
}

}  // namespace

bool coarse_gcr_group_ok(const LevelGeom& G, const CoarseOp& C, int nb) {
  // pairs of complex numbers are loaded as 16 bytes: Nc = 2 Nv is even
  if (nb < 1 || nb > kMaxSys || C.nc % 2 || C.nc > 64 || !C.A.get()) return false;
  return make_plan(G, C.nc, nb).chunk >= 1;
}

void coarse_gcr_group_solve(const std::vector<CoarseSystem>& sys, CoarseGCRBuffers& B, int m, int maxit, int* flags,
                            cudaStream_t s) {
  const int nb = (int)sys.size();
  if (nb < 1) raise(MG_ERR_ARG, "no coarse systems");
  const LevelGeom& G = *sys[0].G;
  const CoarseOp& C = *sys[0].C;
  if (m > kMaxRestart) raise(MG_ERR_ARG, "coarse restart too long for the persistent solver");
  if (!coarse_gcr_group_ok(G, C, nb)) raise(MG_ERR_STATE, "grouped coarse solve not applicable to this level");
  const int nc = C.nc, NS = ns_for(nb);
  const Plan p = make_plan(G, nc, nb);
  GArgs a;
  std::memset(&a, 0, sizeof(a));
  SysPtrs pre{}, post{};
  a.nc = nc;
  a.half = G.half;
  a.rows_sites = G.eo ? G.half : G.nsites;
  a.m = m;
  a.maxit = maxit;
  a.nb = nb;
  a.ips = p.ips;
  a.items = p.items;
  a.chunk = p.chunk;
  const size_t n = (size_t)a.rows_sites * nc;
  B.grow(B.gp_v, sizeof(float2) * n * nb * 5);
  B.grow(B.gp_W, sizeof(float2) * n * nb * (size_t)m);
  B.grow(B.gp_R, sizeof(float2) * n * nb * (size_t)m);
  B.grow(B.gp_part, sizeof(float2) * (size_t)nb * kSlots * p.grid);
  B.grow(B.gp_sync, 512 + sizeof(float2) * (kMaxSys * (size_t)(kSlots + 2 * kMaxRestart + kMaxRestart * kMaxRestart)));
  float2* v = B.gp_v.as<float2>();
  a.y = v;
  a.r = v + n * nb;
  a.br = v + 2 * n * nb;
  a.tb = v + 3 * n * nb;
  a.t = v + 4 * n * nb;
  a.W = B.gp_W.as<float2>();
  a.R = B.gp_R.as<float2>();
  a.part = B.gp_part.as<float2>();
  unsigned char* sync = B.gp_sync.as<unsigned char>();
  a.bar = reinterpret_cast<unsigned*>(sync);
  a.abort = reinterpret_cast<int*>(sync + 128);
  a.tot = reinterpret_cast<float2*>(sync + 512);
  a.ag = a.tot + kMaxSys * kSlots;
  a.beta = a.ag + 2 * kMaxSys * kMaxRestart;
  a.nbr = G.d_nbr.as<int>();
  a.Y = static_cast<const unsigned char*>(C.Y.get());
  a.Ys = C.Yscale.as<float>();
  a.A = static_cast<const unsigned char*>(C.A.get());
  a.flags = flags;
  for (int q = 0; q < nb; q++) {
    if (sys[q].G != sys[0].G || sys[q].C != sys[0].C) raise(MG_ERR_ARG, "grouped coarse systems share one lattice");
    a.tol_rel[q] = (float)sys[q].tol_rel;
    a.b[q] = reinterpret_cast<const float2*>(sys[q].b);
    a.x[q] = reinterpret_cast<float2*>(sys[q].x);
    a.iters[q] = sys[q].iters;
    pre.in[q] = a.b[q];
    pre.out[q] = a.tb + n * q;
    post.in[q] = a.y + n * q;
    post.out[q] = a.x[q];
  }
  MG_CUDA(cudaMemsetAsync(sync, 0, 512, s));
  const size_t smul = sizeof(float2) * (size_t)nb * nc;
  const float2* Xinv = C.Xinv.as<float2>();
  if (G.eo) {   // X_o^{-1} b_o
    k_site_mul_systems<<<G.nsites - G.half, kThreads, smul, s>>>(nc, nb, G.half, 0, G.half, Xinv, pre);
    MG_LAUNCH();
  }
  const void* kern = kernel_for(G.eo, C.store, NS);
  int per = 0, dev = 0, sms = 0;
  MG_CUDA(cudaGetDevice(&dev));
  MG_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  MG_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem));
  MG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, kThreads, p.smem));
  if (per < 1 || p.grid > per * sms) raise(MG_ERR_CUDA, "grouped coarse GCR cannot be resident");
  void* params[] = {&a};
  MG_CUDA(cudaLaunchCooperativeKernel(kern, dim3(p.grid), dim3(kThreads), params, p.smem, s));
  MG_LAUNCH();
  if (G.eo) {   // x_e = X_e^{-1} y_e
    k_site_mul_systems<<<G.half, kThreads, smul, s>>>(nc, nb, 0, 0, 0, Xinv, post);
    MG_LAUNCH();
  }
}

}  // namespace mg
