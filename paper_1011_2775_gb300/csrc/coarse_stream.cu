// The coarsest-level GCR of an even-odd coarse lattice with its links
// streamed through shared memory.
//
// Same method as coarse_gcr.cu (section "Implementation": unpreconditioned
// GCR on the coarsest lattice to a relative residual tolerance; section
// "Red-black preconditioning": the reduced even-odd system
// D_r = 1 - Y_eo X_o^{-1} Y_oe X_e^{-1}), arranged for the GB300 memory
// system:
//
//  * Work items are row blocks of one site's link matrix (rows x 8 Nc):
//    phase A uses the folded odd-site links X_o^{-1} Y_d X^{-1}(o + d) (FP32),
//    phase B the even-site links Y_eo in their storage format.  Every block
//    owns a fixed, contiguous range of A items and of B items, and warp w of
//    the block takes every W-th item of each range (W = 16 or 8 warps).
//  * The links do not change during the solve, so the order in which a warp
//    consumes them is known in advance: its B items (for b_r), then its A
//    items and B items once per operator application.  Each warp keeps two
//    shared-memory stages filled along its sequence with bulk asynchronous
//    copies (cp.async.bulk, completion on one mbarrier per stage), so the
//    warps stream and compute independently and the links of the next phase
//    arrive while the block waits at a grid barrier.  A warp computes all
//    rows of its item: every lane strides along the row, the gathered vector
//    element is loaded once for all rows, and one transposing shuffle
//    reduction finishes an item's rows (two, four or eight of them).
//  * The element-wise work belongs to the block that computed those rows in
//    phase B, so the Gram-Schmidt dots follow phase B without a barrier:
//    one iteration is phase A | barrier | phase B + dots | barrier |
//    coefficients, update, ||r||^2 | barrier.  The norm of the orthogonalised
//    w comes from Pythagoras (the w_j are orthonormal), with an exact second
//    reduction when that subtraction loses more than three digits; <w', r>
//    = <w, r> / gamma because r is orthogonal to the w_j.  The block's slice
//    of the Krylov vectors w_j stays in shared memory when it is small.
//  * Every inner product is reduced deterministically (per-block double-float
//    partials summed in the same order by every block), so all blocks take
//    identical decisions and the result is reproducible bit for bit.
//  * Every wait (mbarrier, grid barrier) is bounded in time; a block that
//    times out raises an abort flag that releases the others, sets
//    FLAG_TIMEOUT and the kernel returns after its copies in flight land.
//
// The site-local parts around it -- t_o = X_o^{-1} b_o before and x_e = X_e^{-1} y_e
// after -- are separate launches.  The closing true residual has formed A y on
// the odd sites, so x_o = X_o^{-1} (b_o - Y_oe x_e) = t_o - A y is written there
// instead of by another pass over the links (17 us of a 16^3x32 solve, 112 of
// 427 us at 24^3x48 with bf16 links).
//
// Measured (16^3x32, 4^4 blocks, Nc = 48, 256 reduced sites, 35 iterations):
// 817 us per solve with 256 threads, neighbour indices read for every gather,
// the coefficients formed before the sums, divisions and a switch over the rows
// of every item, and r and w read back from global memory; 618 us here.  Of the
// 38k cycles of an iteration the stencil passes take 6.6k each (shared-memory
// port: every link byte is written and read there, every gathered vector read
// once per two rows), the gathers 1.5k each, the barriers 9k, inner products,
// totals, coefficients and update 12k.  24^3x48 with bf16 links: 427 -> 269 us;
// the links come from HBM and phase A runs at its rate (191 MB in 28.6 us).
// On a lattice with an odd extent the same loop applies D_hat = [Y_0 .. Y_7 | X]
// on all sites: 3^3x6, Nc = 48: 112 us on the grouped kernel with one system, 67 here.
#include <algorithm>
#include <cstring>

#include "async_copy.cuh"
#include "dfloat.cuh"
#include "coarse.h"
#include "coarse_dev.cuh"

namespace mg {

namespace {

constexpr int kStagesPerWarp = 2;
constexpr int kMaxRows = 8;        // rows of one item (16 accumulators per lane)
constexpr int kMaxGroups = 8;      // thread groups sharing the sum over j of the Gram-Schmidt update
constexpr int kMaxRestart = 64;
// reduction slots: [0, 2 kMaxRestart) <w_j, w>; then ||w||^2, Re/Im <w, r>;
// ||r||^2; ||b||^2 / true residual; the exact ||w'||^2, Re/Im <w', r>
constexpr int RA = 0;
constexpr int RB = 2 * kMaxRestart;
constexpr int RC = RB + 3;
constexpr int RD = RC + 1;
constexpr int RE = RD + 1;
constexpr int kNR = RE + 3;

struct SArgs {
  int nc, half, m, maxit;     // half: sites of the solved system (all of them on an odd extent)
  int rowsA, rowsB, ipsA, ipsB, NA, NB, eszB;
  int stage_bytes, gmax, wsm_ld;   // wsm_ld > 0: the w_j slice in shared memory, leading dimension
  int esm;                         // > 0: r and w of the owned rows in shared memory, their capacity
  double tol_rel;
  const int* nbr;
  const unsigned char* Y;     // even-site links [e][nc][8][nc], storage format; odd extents: [s][nc][9][nc], FP32
  const float* Ys;            // their tile scales [e][8]
  const unsigned char* Af;    // folded odd-site links [o - half][nc][8][nc], FP32
  const float2* b;            // full right-hand side
  const float2* to;           // full: the odd part holds X_o^{-1} b_o
  float2* x;                  // full solution: the odd half is written here
  float2* y;                  // half: GCR iterate
  float2* r;                  // half: residual
  float2* br;                 // half: reduced right-hand side
  float2* tB;                 // full: the odd part holds the phase-A outputs
  float2* w;                  // half: D_r r, when the owned rows are not in shared memory
  float2* W;                  // [m][half nc] (when the slice is not in shared memory)
  float2* Z;                  // [m][half nc]
  float2* partials;           // [kNR][grid] double-float partial sums
  long long* iters;
  int* flags;
  unsigned* bar;              // grid barrier counter (0 at launch)
  int* abort;
};

// first element (of the half vector) of item i: site i / ips, rows from (i % ips) rows
__device__ __forceinline__ size_t item_elem(int i, int ips, int rows, int nc) {
  return (size_t)(i / ips) * nc + (size_t)(i % ips) * rows;
}

// A block's items [i0, i1) of one phase: this warp's are i0 + wid, i0 + wid + W,
// ...; sl and rem: site (from the block's first) and item of the site of the
// warp's first item, dq and dr their steps (no division per item).
struct Items {
  int i0, i1, ips, sl, rem, dq, dr;
  __device__ Items(int b, int G, int n, int ips_, int W, int wid) : ips(ips_) {
    i0 = (int)((long long)b * n / G);
    i1 = (int)((long long)(b + 1) * n / G);
    const int first = i0 + wid;
    sl = first / ips - i0 / ips;
    rem = first % ips;
    dq = W / ips;
    dr = W % ips;
  }
  __device__ int site0() const { return i0 / ips; }
  __device__ int sites() const { return i1 > i0 ? (i1 - 1) / ips - i0 / ips + 1 : 0; }
};

// rows of a phase-B item: the bytes of R rows of phase A
__host__ __device__ constexpr int rows_b(int st, int R) { return st == kStF32 || R == 0 ? R : 2 * R < kMaxRows ? 2 * R : kMaxRows; }

// Per-warp state of the link stream: items consumed, and the next one to copy.
struct Stream {
  unsigned char* ring;   // this warp's stages
  uint64_t* full;
  unsigned t;            // items consumed
  int kind, it;          // next item to copy: 0 A, 1 B
};

// lane 0: bulk copy of the next item of the sequence into stage `slot`, and on
// to the one after it (the warp's B items for b_r, then A and B alternately)
template <int W, int ND>
__device__ __forceinline__ void issue(const SArgs& a, Stream& st, const Items& A, const Items& B, unsigned slot) {
  const int wid = threadIdx.x >> 5;
  for (int tries = 0; tries < 2 && st.it >= (st.kind ? B.i1 : A.i1); tries++) {   // a phase without items is passed over
    st.kind ^= 1;
    st.it = (st.kind ? B.i0 : A.i0) + wid;
  }
  if (st.it >= (st.kind ? B.i1 : A.i1)) return;
  const int nc = a.nc, rows = st.kind ? a.rowsB : a.rowsA, ips = st.kind ? a.ipsB : a.ipsA;
  size_t row0 = (size_t)st.it * rows;
  int nr = rows;
  if (ips * rows != nc) {   // the last item of a site is short
    const int s = st.it / ips, r0 = (st.it - s * ips) * rows;
    row0 = (size_t)s * nc + r0;
    nr = min(rows, nc - r0);
  }
  const unsigned per = (unsigned)ND * nc * (st.kind ? a.eszB : 8);
  const unsigned bytes = nr * per;
  mbar_arrive_expect_tx(&st.full[slot], bytes);
  bulk_copy_g2s(st.ring + (size_t)slot * a.stage_bytes, (st.kind ? a.Y : a.Af) + row0 * per, bytes, &st.full[slot]);
  st.it += W;
}

// Gathers the vectors of the block's `ns` sites of a phase: for each site, the
// 8 neighbours' nc components of `in` (neighbour indices in shared memory),
// times the tile scale of Y (phase B).  A warp takes (site, direction) pairs,
// 16 bytes per lane, the loads of kGather pairs in flight together: one L2
// round trip for a block of up to eight sites.
constexpr int kGather = 4;
template <int kWarps, int ND>
__device__ __forceinline__ void gather(int nc, int ns, const int* nbr, const float* scale, const float2* in, float2* gv) {
  const int nc2 = nc >> 1, np = ND * ns, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float4* g4 = reinterpret_cast<float4*>(gv);
  for (int p0 = w; p0 < np; p0 += kGather * kWarps)
    for (int q = lane; q < nc2; q += 32) {
      float4 v[kGather];
#pragma unroll
      for (int u = 0; u < kGather; u++) {
        const int p = min(p0 + u * kWarps, np - 1);
        v[u] = __ldcg(reinterpret_cast<const float4*>(in + (size_t)nbr[p] * nc) + q);
      }
#pragma unroll
      for (int u = 0; u < kGather; u++) {
        const int p = p0 + u * kWarps;
        if (p >= np) break;
        const float c = scale ? scale[p] : 1.f;
        g4[(size_t)p * nc2 + q] = make_float4(c * v[u].x, c * v[u].y, c * v[u].z, c * v[u].w);
      }
    }
  __syncthreads();
}

// out[row] = sum_k L[row][k] v[k] for the NR rows of a staged item (row-major,
// K complex per row, storage format ST).  Every lane strides along the rows
// two float4 steps at a time, loading the vector element once for all rows.
// Returns true on the lane that holds row `row`'s {re, im} in `res`.
template <int ST, int NR>
__device__ __forceinline__ bool item_rows(const unsigned char* stage, int K, const float2* v, float2& res, int& row) {
  constexpr int V = NR <= 1 ? 2 : NR <= 2 ? 4 : NR <= 4 ? 8 : 16;
  constexpr int SH = V == 2 ? 4 : V == 4 ? 3 : V == 8 ? 2 : 1;   // log2(32 / V)
  const float4* v4 = reinterpret_cast<const float4*>(v);
  const int lane = threadIdx.x & 31;
  const int K2 = K >> 1;
  float acc[V];
#pragma unroll
  for (int i = 0; i < V; i++) acc[i] = 0.f;
  auto step = [&](int q) {
    const float4 x = v4[q];
#pragma unroll
    for (int r = 0; r < NR; r++) {
      float4 m;
      if constexpr (ST == kStF32)
        m = reinterpret_cast<const float4*>(stage)[(size_t)r * K2 + q];
      else
        m = LinkPair<ST>::decode(reinterpret_cast<const uint2*>(stage)[(size_t)r * K2 + q]);
      acc[2 * r] = fmaf(m.x, x.x, acc[2 * r]);
      acc[2 * r] = fmaf(-m.y, x.y, acc[2 * r]);
      acc[2 * r] = fmaf(m.z, x.z, acc[2 * r]);
      acc[2 * r] = fmaf(-m.w, x.w, acc[2 * r]);
      acc[2 * r + 1] = fmaf(m.x, x.y, acc[2 * r + 1]);
      acc[2 * r + 1] = fmaf(m.y, x.x, acc[2 * r + 1]);
      acc[2 * r + 1] = fmaf(m.z, x.w, acc[2 * r + 1]);
      acc[2 * r + 1] = fmaf(m.w, x.z, acc[2 * r + 1]);
    }
  };
#pragma unroll 3
  for (int q = lane; q < K2; q += 32) step(q);
  const float t = warp_transpose_sum<V>(acc);                       // lane l: value (l >> SH) & (V - 1)
  const float im = __shfl_down_sync(0xffffffffu, t, 1 << SH);  // value 2 row + 1
  res = make_float2(t, im);
  row = lane >> (SH + 1);
  return (lane & ((2 << SH) - 1)) == 0 && row < NR;
}

// One phase of this warp's items: waits for each staged item, computes its
// rows, hands them to epi(element from the block's first site, row value) and
// refills the stage two items ahead.  false on a timeout (uniform in the block).
template <int ST, int NR, int W, int ND, typename Epi>
__device__ __forceinline__ bool run_items(const SArgs& a, Stream& st, const Items& A, const Items& B, const Items& g,
                                          const float2* gv, Epi epi, int* s_fail) {
  const int nc = a.nc, K = ND * nc, lane = threadIdx.x & 31;
  int sl = g.sl, rem = g.rem;
  for (int it = g.i0 + (threadIdx.x >> 5); it < g.i1; it += W) {
    const unsigned slot = st.t % kStagesPerWarp;
    if (!mbar_wait(&st.full[slot], (st.t / kStagesPerWarp) & 1u)) {
      atomicExch(s_fail, 1);
      break;
    }
    const int r0 = rem * NR;
    float2 res;
    int row;   // rows past the site's last are not copied; what their sums hold is dropped
    const bool mine = item_rows<ST, NR>(st.ring + (size_t)slot * a.stage_bytes, K, gv + (size_t)sl * K, res, row);
    __syncwarp();
    if (lane == 0) issue<W, ND>(a, st, A, B, slot);
    if (mine && r0 + row < nc) epi(sl * nc + r0 + row, res);
    st.t++;
    sl += g.dq;
    rem += g.dr;
    if (rem >= g.ips) {
      rem -= g.ips;
      sl++;
    }
  }
  __syncthreads();
  return *(volatile int*)s_fail == 0;
}

// block partial sums of nq <= 4 per-thread float values v[q]: one transposed
// warp reduction for the four, then warp q adds the warps' sums of value q;
// partials[q0 + q][block]
template <int kWarps>
__device__ __forceinline__ void block_partials(const SArgs& a, const float* v, int nq, int q0, df* sred) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  df t[4];
#pragma unroll
  for (int q = 0; q < 4; q++) t[q] = df_of(q < nq ? v[q] : 0.f);
  const df ws = warp_transpose_sum<4>(t);   // lane l: value l >> 3
  if ((lane & 7) == 0) sred[(lane >> 3) * kWarps + wid] = ws;
  __syncthreads();
  if (wid < nq) {
    const df s = df_wsum(lane < kWarps ? sred[wid * kWarps + lane] : df_of(0.f));
    if (lane == 0) a.partials[(size_t)(q0 + wid) * gridDim.x + blockIdx.x] = make_float2(s.h, s.l);
  }
  __syncthreads();
}

// totals of slots [q0, q0 + nq) after a grid barrier, identical in every
// block.  Warp w sums slots w, w + kWarps, ...; each round issues the loads of U
// slots (up to kTotG / 32 per lane and slot) before adding any, so that a
// round costs one L2 round trip; the U sums leave the warp through one
// transposing reduction.
constexpr int kTotG = 160;   // grids up to this size take the one-pass path
template <int U, int kWarps>
__device__ __forceinline__ void totals_rounds(const SArgs& a, int q0, int nq, df* out) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int G = gridDim.x;
  for (int qb = wid; qb < nq; qb += U * kWarps) {
    float2 t[U][kTotG / 32];
#pragma unroll
    for (int u = 0; u < U; u++) {
      const int q = qb + u * kWarps;
      const float2* p = a.partials + (size_t)(q0 + (q < nq ? q : 0)) * G;
#pragma unroll
      for (int i = 0; i < kTotG / 32; i++) {
        const int g = lane + 32 * i;
        t[u][i] = (q < nq && g < G) ? __ldcg(p + g) : make_float2(0.f, 0.f);
      }
    }
    df sv[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
      sv[u] = df{t[u][0].x, t[u][0].y};
#pragma unroll
      for (int i = 1; i < kTotG / 32; i++) sv[u] = df_add(sv[u], df{t[u][i].x, t[u][i].y});
    }
    const df s = warp_transpose_sum<U>(sv);   // lane l: slot qb + l / (32 / U) * kWarps
    const int q = qb + lane / (32 / U) * kWarps;
    if (lane % (32 / U) == 0 && q < nq) out[q] = s;
  }
}
template <int kWarps>
__device__ __forceinline__ void grid_totals(const SArgs& a, int q0, int nq, df* out) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int G = gridDim.x;
  if (G <= kTotG) {
    if (nq <= kWarps)
      totals_rounds<1, kWarps>(a, q0, nq, out);
    else if (nq <= 4 * kWarps)
      totals_rounds<4, kWarps>(a, q0, nq, out);
    else
      totals_rounds<8, kWarps>(a, q0, nq, out);
  } else {
    for (int q = wid; q < nq; q += kWarps) {
      const float2* p = a.partials + (size_t)(q0 + q) * G;
      df s = df_of(0.f);
      for (int g = lane; g < G; g += 32) {
        const float2 x = __ldcg(p + g);
        s = df_add(s, df{x.x, x.y});
      }
      s = df_wsum(s);
      if (lane == 0) out[q] = s;
    }
  }
  __syncthreads();
}

// What the next pass over the links is for: b_r at the start, w = D_r r of an
// iteration, or the true residual that closes a restart cycle.  One loop and
// one copy of the two stencil phases serve all three: the code of an iteration
// is fetched again every time round.
enum { M_INIT, M_ITER, M_CLOSE };

// W warps, R rows per item of phase A (phase B, 16-bit links: 2 R).  On a
// lattice with an odd extent (EO false) there is phase B alone, D_hat v with the
// links [Y_0 .. Y_7 | X] of all sites.
template <int ST, int W, int R, bool EO>
__global__ void __launch_bounds__(32 * W, 1) k_coarse_gcr_stream(const __grid_constant__ SArgs a) {
  constexpr int kThreads = 32 * W, kUpdThreads = kThreads - 32;   // warp 0 forms the coefficients meanwhile
  constexpr int RB_ = rows_b(ST, R), ND = EO ? 8 : 9;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t full[W * kStagesPerWarp];
  __shared__ float s_coef[4];              // 1/gamma, Re alpha, Im alpha, exact flag
  __shared__ int s_fail;
  const int nc = a.nc, K = ND * nc, m = a.m;
  const int G = gridDim.x, bid = blockIdx.x;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  float2* gv = reinterpret_cast<float2*>(smem + (size_t)W * kStagesPerWarp * a.stage_bytes);
  float2* upd = gv + (size_t)a.gmax * K;                               // [2][kThreads] update partial sums
  float2* wsm = upd + 2 * kThreads;                                    // [m][wsm_ld] when used
  float2* esm = wsm + (size_t)m * a.wsm_ld;                            // [2][esm] when used
  df* sred = reinterpret_cast<df*>(esm + 2 * (size_t)a.esm);           // [4][W]
  df* tot = sred + 4 * W;                                              // [kNR]
  int* nbA = reinterpret_cast<int*>(tot + kNR);                        // [gmax][8] neighbours of the A sites,
  int* nbB = nbA + 8 * a.gmax;                                         // [gmax][ND] of the B sites,
  float* scB = reinterpret_cast<float*>(nbB + 9 * a.gmax);             // and the tile scales of the B sites

  const Items A(bid, G, a.NA, a.ipsA, W, wid), B(bid, G, a.NB, a.ipsB, W, wid);
  Stream st;
  st.ring = smem + (size_t)wid * kStagesPerWarp * a.stage_bytes;
  st.full = full + wid * kStagesPerWarp;
  st.t = 0;
  st.kind = 1;
  st.it = B.i0 + wid;
  const int sA = A.site0(), nA = A.sites(), sB = B.site0(), nB = B.sites();
  const size_t E0 = item_elem(B.i0, a.ipsB, RB_, nc);
  const size_t E1 = B.i1 == a.NB ? (size_t)a.half * nc : item_elem(B.i1, a.ipsB, RB_, nc);
  const int E = (int)(E1 - E0), offB = (int)(E0 - (size_t)sB * nc);
  const size_t n = (size_t)a.half * nc, oA = ((size_t)a.half + sA) * nc;
  // the block's slices of w_j and z_j: element e at Wj(j)[e - E0], Zj(j)[e - E0]
  float2* const wbase = a.wsm_ld > 0 ? wsm : a.W + E0;
  const size_t wld = a.wsm_ld > 0 ? (size_t)a.wsm_ld : n;
  auto Wj = [&](int j) { return wbase + (size_t)j * wld; };
  auto Zj = [&](int j) { return a.Z + (size_t)j * n + E0; };
  // r and w = D_r r on the owned rows (r also in global memory, for the gathers)
  float2* const rs = a.esm > 0 ? esm : a.r + E0;
  float2* const ws = a.esm > 0 ? esm + a.esm : a.w + E0;
  // the j sums of the Gram-Schmidt update are split over ngrp groups of the
  // threads of warps 1 .. when the slice has at most one element per thread
  const int ngrp = (E > 0 && E <= kUpdThreads) ? min(kUpdThreads / E, kMaxGroups) : 0;
  unsigned target = 0;
  bool ok = true;
  float v[4];

  if (threadIdx.x == 0) {
    for (int s = 0; s < W * kStagesPerWarp; s++) mbar_init(&full[s], 1);
    mbar_fence_init();
    s_fail = 0;
  }
  for (int i = threadIdx.x; i < 8 * nA; i += kThreads) nbA[i] = a.nbr[(size_t)(a.half + sA) * 8 + i];
  if (EO) {
    for (int i = threadIdx.x; i < 8 * nB; i += kThreads) {
      nbB[i] = a.nbr[(size_t)sB * 8 + i];
      scB[i] = a.Ys[(size_t)sB * 8 + i];
    }
  } else {
    for (int i = threadIdx.x; i < 9 * nB; i += kThreads) {
      const int sl = i / 9, d = i - 9 * sl;
      nbB[i] = d < 8 ? a.nbr[(size_t)(sB + sl) * 8 + d] : sB + sl;
    }
  }
  __syncthreads();
  if (lane == 0)
    for (unsigned p = 0; p < kStagesPerWarp; p++) issue<W, ND>(a, st, A, B, p);

  int mode = M_INIT, k = 0;
  long long its = 0;
  df tol2 = df_of(0.f);
  while (true) {
    if (EO && mode != M_INIT) {
      // phase A: A v on the odd sites; in the closing pass v = y, and the odd
      // half of the solution is x_o = X_o^{-1} b_o - A y
      gather<W, ND>(nc, nA, nbA, nullptr, mode == M_ITER ? a.r : a.y, gv);
      ok = run_items<kStF32, R, W, ND>(a, st, A, B, A, gv, [&](int e, float2 u) {
        a.tB[oA + e] = u;
        if (mode == M_CLOSE) {
          const float2 o = a.to[oA + e];
          a.x[oA + e] = make_float2(o.x - u.x, o.y - u.y);
        }
      }, &s_fail);
      if (!ok || !(ok = grid_barrier(a.bar, a.abort, target))) break;
    }
    // phase B on the even sites: w = r - Y_eo t, without r outside the iterations
    // (or w = D_hat v on all sites)
    if (EO || mode != M_INIT) {
      if (EO)
        gather<W, ND>(nc, nB, nbB, scB, mode == M_INIT ? a.to : a.tB, gv);
      else
        gather<W, ND>(nc, nB, nbB, nullptr, mode == M_ITER ? a.r : a.y, gv);
      ok = run_items<ST, RB_, W, ND>(a, st, A, B, B, gv, [&](int e, float2 u) {
        const float2 o = EO && mode == M_ITER ? rs[e - offB] : make_float2(0.f, 0.f);
        ws[e - offB] = EO ? make_float2(o.x - u.x, o.y - u.y) : u;
      }, &s_fail);
      if (!ok) break;
    }
    if (mode != M_ITER) {
      // b_r = b_e - Y_eo X_o^{-1} b_o, r = b_r, y = 0; or the true r = b_r - D_r y
      v[0] = v[1] = 0.f;
      for (int e = threadIdx.x; e < E; e += kThreads) {
        float2 rr, u = make_float2(0.f, 0.f);
        if (EO || mode != M_INIT) u = ws[e];
        if (mode == M_INIT) {
          const float2 bb = a.b[E0 + e];
          rr = make_float2(bb.x + u.x, bb.y + u.y);
          if (EO) a.br[E0 + e] = rr;
          a.y[E0 + e] = make_float2(0.f, 0.f);
        } else if (!EO) {
          const float2 bb = a.b[E0 + e];
          rr = make_float2(bb.x - u.x, bb.y - u.y);
        } else {
          const float2 bb = a.br[E0 + e], yy = a.y[E0 + e];
          rr = make_float2(bb.x - (yy.x + u.x), bb.y - (yy.y + u.y));
        }
        rs[e] = rr;
        a.r[E0 + e] = rr;
        v[0] = fmaf(rr.x, rr.x, fmaf(rr.y, rr.y, v[0]));
      }
      if (mode == M_INIT) {   // ||b||^2 over the full right-hand side (any partition of it)
        const size_t nf = EO ? 2 * n : n, cf = (nf + G - 1) / G;
        const size_t f0 = (size_t)bid * cf, f1 = f0 + cf < nf ? f0 + cf : nf;
        for (size_t e = f0 + threadIdx.x; e < f1; e += kThreads) {
          const float2 q = a.b[e];
          v[1] = fmaf(q.x, q.x, fmaf(q.y, q.y, v[1]));
        }
      }
      const int nq = mode == M_INIT ? 2 : 1;
      block_partials<W>(a, v, nq, RC, sred);
      if (!(ok = grid_barrier(a.bar, a.abort, target))) break;
      grid_totals<W>(a, RC, nq, tot + RC);   // ||r||^2 restarts the running norm
      if (mode == M_INIT) {
        const df tr = df_of((float)a.tol_rel);
        tol2 = df_mul(df_mul(tr, tr), tot[RD]);
        if (!(tot[RD].h > 0.f) && tot[RC].h == tot[RC].h) break;
      } else if (tot[RC].h <= tol2.h) {
        break;
      }
      if (!(tot[RC].h == tot[RC].h)) {
        if (bid == 0 && threadIdx.x == 0) atomicExch(&a.flags[FLAG_NAN], 1);
        break;
      }
      if (its >= a.maxit) break;
      mode = M_ITER;
      k = 0;
      continue;
    }
    float2* wk = Wj(k);
    // beta_j = <w_j, w> (warp wid owns j = wid + W u, u < 4), ||w||^2, <w, r>
    for (int jb = wid; jb < k; jb += 4 * W) {
      float re[4] = {0.f, 0.f, 0.f, 0.f}, im[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
      for (int e = lane; e < E; e += 32) {
        const float2 x = ws[e];
#pragma unroll
        for (int u = 0; u < 4; u++) {
          const int j = jb + u * W;
          const float2 p = j < k ? Wj(j)[e] : make_float2(0.f, 0.f);
          re[u] = fmaf(p.x, x.x, fmaf(p.y, x.y, re[u]));
          im[u] = fmaf(p.x, x.y, fmaf(-p.y, x.x, im[u]));
        }
      }
      df sv[8];
#pragma unroll
      for (int u = 0; u < 4; u++) {
        sv[2 * u] = df_of(re[u]);
        sv[2 * u + 1] = df_of(im[u]);
      }
      const df sr = warp_transpose_sum<8>(sv);   // lane l: sum (l >> 2) = 2 u + {re, im}
      const int j = jb + (lane >> 3) * W;
      if ((lane & 3) == 0 && j < k) a.partials[(size_t)(RA + 2 * j + ((lane >> 2) & 1)) * G + bid] = make_float2(sr.h, sr.l);
    }
    v[0] = v[1] = v[2] = 0.f;
    for (int e = threadIdx.x; e < E; e += kThreads) {
      const float2 x = ws[e], rr = rs[e];
      v[0] = fmaf(x.x, x.x, fmaf(x.y, x.y, v[0]));
      v[1] = fmaf(x.x, rr.x, fmaf(x.y, rr.y, v[1]));
      v[2] = fmaf(x.x, rr.y, fmaf(-x.y, rr.x, v[2]));
    }
    block_partials<W>(a, v, 3, RA + 2 * k, sred);   // after the beta slots: one pass reads all of them
    if (!(ok = grid_barrier(a.bar, a.abort, target))) break;
    grid_totals<W>(a, RA, 2 * k + 3, tot);
    // warp 0: sum_j |beta_j|^2 and the coefficients; the other warps meanwhile
    // S_w = sum_j beta_j w_j, S_z = sum_j beta_j z_j on the owned rows
    auto beta = [&](int j) {
      return make_float2(tot[2 * j].h + tot[2 * j].l, tot[2 * j + 1].h + tot[2 * j + 1].l);
    };
    // gamma = ||w''||, alpha = <w'', r> / gamma; with w_k = w'' / gamma of
    // unit norm, ||r - alpha w_k||^2 = ||r||^2 - |alpha|^2 (the running norm)
    auto coefficients = [&](df g2, df wr, df wi) {
      const df g = df_sqrt(g2);
      const bool gz = !(g.h > 0.f);
      s_coef[0] = gz ? 1.f : 1.f / g.h;
      const df ar = gz ? wr : df_div(wr, g);
      const df ai = gz ? wi : df_div(wi, g);
      s_coef[1] = ar.h + ar.l;
      s_coef[2] = ai.h + ai.l;
      if (!(g2.h == g2.h)) {   // NaN in w: the running norm carries it to the test below
        tot[RC] = g2;
      } else if (!gz) {
        const df rn = df_add(tot[RC], df_neg(df_add(df_mul(ar, ar), df_mul(ai, ai))));
        tot[RC] = rn.h > 0.f || !(rn.h == rn.h) ? rn : df_of(0.f);
      }
    };
    if (wid == 0) {
      df bb = df_of(0.f);
      for (int j = lane; j < k; j += 32) {
        bb = df_add(bb, df_mul(tot[2 * j], tot[2 * j]));
        bb = df_add(bb, df_mul(tot[2 * j + 1], tot[2 * j + 1]));
      }
      bb = df_wsum(bb);
      if (lane == 0) {
        const df ww = tot[2 * k], g2 = df_add(ww, df_neg(bb));
        const bool fine = g2.h > 1e-3f * ww.h;   // otherwise Pythagoras lost more than three digits
        s_coef[3] = fine ? 0.f : 1.f;
        if (fine) coefficients(g2, tot[2 * k + 1], tot[2 * k + 2]);
      }
    } else if (ngrp) {
      const int t = threadIdx.x - 32, gi = t / E, ei = t - gi * E;
      if (gi < ngrp) {
        float swr = 0.f, swi = 0.f, szr = 0.f, szi = 0.f;
#pragma unroll 8
        for (int j = gi; j < k; j += ngrp) {
          const float2 bj = beta(j);
          const float2 p = Wj(j)[ei], q = Zj(j)[ei];
          swr = fmaf(bj.x, p.x, fmaf(-bj.y, p.y, swr));
          swi = fmaf(bj.x, p.y, fmaf(bj.y, p.x, swi));
          szr = fmaf(bj.x, q.x, fmaf(-bj.y, q.y, szr));
          szi = fmaf(bj.x, q.y, fmaf(bj.y, q.x, szi));
        }
        upd[gi * E + ei] = make_float2(swr, swi);
        upd[kThreads + gi * E + ei] = make_float2(szr, szi);
      }
    }
    __syncthreads();
    const bool exact = s_coef[3] != 0.f;
    // w'' = w - S_w
    auto w_orth = [&](int ei) {
      float2 x = ws[ei];
      if (ngrp) {
        for (int g = 0; g < ngrp; g++) {
          const float2 u = upd[g * E + ei];
          x.x -= u.x;
          x.y -= u.y;
        }
      } else {
#pragma unroll 4
        for (int j = 0; j < k; j++) {
          const float2 bj = beta(j), p = Wj(j)[ei];
          x.x -= bj.x * p.x - bj.y * p.y;
          x.y -= bj.x * p.y + bj.y * p.x;
        }
      }
      return x;
    };
    if (exact) {  // uniform: every block took the same decision from the same totals
      v[0] = v[1] = v[2] = 0.f;
      for (int ei = threadIdx.x; ei < E; ei += kThreads) {
        const float2 x = w_orth(ei), rr = rs[ei];
        v[0] = fmaf(x.x, x.x, fmaf(x.y, x.y, v[0]));
        v[1] = fmaf(x.x, rr.x, fmaf(x.y, rr.y, v[1]));
        v[2] = fmaf(x.x, rr.y, fmaf(-x.y, rr.x, v[2]));
      }
      block_partials<W>(a, v, 3, RE, sred);
      if (!(ok = grid_barrier(a.bar, a.abort, target))) break;
      grid_totals<W>(a, RE, 3, tot + RB);   // the exact ||w''||^2, <w'', r> replace the estimates
      if (threadIdx.x == 0) coefficients(tot[RB], tot[RB + 1], tot[RB + 2]);
      __syncthreads();
    }
    // w_k = w'' / gamma, z_k = (r - S_z) / gamma, y += alpha z_k, r -= alpha w_k
    const float ig = s_coef[0], far = s_coef[1], fai = s_coef[2];
    v[0] = 0.f;
    for (int ei = threadIdx.x; ei < E; ei += kThreads) {
      const size_t e = E0 + ei;
      float2 x = w_orth(ei);
      x.x *= ig;
      x.y *= ig;
      wk[ei] = x;
      float2 rr = rs[ei];
      float2 z = rr;
      if (ngrp) {
        for (int g = 0; g < ngrp; g++) {
          const float2 u = upd[kThreads + g * E + ei];
          z.x -= u.x;
          z.y -= u.y;
        }
      } else {
#pragma unroll 4
        for (int j = 0; j < k; j++) {
          const float2 bj = beta(j), q = Zj(j)[ei];
          z.x -= bj.x * q.x - bj.y * q.y;
          z.y -= bj.x * q.y + bj.y * q.x;
        }
      }
      z.x *= ig;
      z.y *= ig;
      Zj(k)[ei] = z;
      float2 yy = a.y[e];
      yy.x += far * z.x - fai * z.y;
      yy.y += far * z.y + fai * z.x;
      a.y[e] = yy;
      rr.x -= far * x.x - fai * x.y;
      rr.y -= far * x.y + fai * x.x;
      rs[ei] = rr;
      a.r[e] = rr;
    }
    // r complete on every block before the next phase A reads it
    if (!(ok = grid_barrier(a.bar, a.abort, target))) break;
    k++;
    its++;
    const df rn2 = tot[RC];
    if (!(rn2.h == rn2.h)) {
      if (bid == 0 && threadIdx.x == 0) atomicExch(&a.flags[FLAG_NAN], 1);
      break;
    }
    if (rn2.h <= tol2.h || k == m || its >= a.maxit) mode = M_CLOSE;
  }
  if (EO && ok && its == 0)   // b = 0: y = 0 and x_o = t_o
    for (size_t e = (size_t)bid * kThreads + threadIdx.x; e < n; e += (size_t)G * kThreads) a.x[n + e] = a.to[n + e];
  if (!ok && threadIdx.x == 0) {
    atomicExch(&a.flags[FLAG_TIMEOUT], 1);
    atomicExch(a.abort, 1);
  }
  // drain: the copies this warp issued beyond what it consumed land before exit
  if (lane == 0 && (A.i1 > A.i0 + wid || B.i1 > B.i0 + wid))
    for (unsigned p = st.t; p < st.t + kStagesPerWarp; p++)
      (void)mbar_wait(&st.full[p % kStagesPerWarp], (p / kStagesPerWarp) & 1u);
  if (bid == 0 && threadIdx.x == 0) *a.iters += its;
}

struct Plan {
  int optin, grid, warps, stage_bytes, rowsA, rowsB, ipsA, ipsB, NA, NB, gmax, wsm_ld, esm, emax;
  size_t smem;
};

int pow2_floor(int v) {
  int p = 1;
  while (2 * p <= v) p *= 2;
  return v > 0 ? p : 0;
}

// items, the sites a block's item ranges touch, and the shared memory they need
void plan_items(Plan& p, int sites, int nc, int nd, int store) {
  const int K = nd * nc;
  p.rowsA = pow2_floor(std::min(p.warps == 16 ? kMaxRows : 2, std::min(nc, p.stage_bytes / (K * 8))));
  p.rowsB = rows_b(store == STORE_F32 ? kStF32 : kStF16, p.rowsA);
  p.ipsA = p.rowsA > 0 ? (nc + p.rowsA - 1) / p.rowsA : 0;
  p.ipsB = p.rowsB > 0 ? (nc + p.rowsB - 1) / p.rowsB : 0;
  p.NA = sites * p.ipsA;
  p.NB = sites * p.ipsB;
  p.gmax = 1;
  p.emax = 0;
  const int G = std::min(p.grid, std::min(p.NA, p.NB));
  auto elem = [&](int i) -> long long {   // item_elem of the kernel
    return i == p.NB ? (long long)sites * nc : (long long)(i / p.ipsB) * nc + (long long)(i % p.ipsB) * p.rowsB;
  };
  for (int b = 0; b < G && p.rowsA > 0 && p.rowsB > 0; b++) {
    const int a0 = (int)((long long)b * p.NA / G), a1 = (int)((long long)(b + 1) * p.NA / G);
    const int b0 = (int)((long long)b * p.NB / G), b1 = (int)((long long)(b + 1) * p.NB / G);
    if (a1 > a0) p.gmax = std::max(p.gmax, (a1 - 1) / p.ipsA - a0 / p.ipsA + 1);
    if (b1 > b0) p.gmax = std::max(p.gmax, (b1 - 1) / p.ipsB - b0 / p.ipsB + 1);
    p.emax = std::max(p.emax, (int)(elem(b1) - elem(b0)));
  }
}

Plan plan_warps(const LevelGeom& G, const CoarseOp& C, int grid, int m, int warps) {
  Plan p;
  p.warps = warps;
  const int nc = C.nc, nd = G.eo ? 8 : 9, K = nd * nc, stages = warps * kStagesPerWarp;
  const int sites = G.eo ? G.half : G.nsites, store = G.eo ? C.store : STORE_F32;
  int dev = 0, optin = 0;
  MG_CUDA(cudaGetDevice(&dev));
  MG_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  p.optin = optin;
  const size_t budget = (size_t)optin - 4096;   // static shared memory and slack
  const size_t fixed = sizeof(float2) * (4 * warps + kNR) + sizeof(float2) * 2 * 32 * warps;
  const size_t per_site = sizeof(float2) * K + 25 * sizeof(int);   // gathered vector, neighbours, tile scales
  p.grid = grid;
  // the w_j slice in shared memory only when it is small (a sixteenth of the
  // budget): measured on GB300 at Nc = 48, m = 64, a deeper link ring gains
  // more than shared-memory Gram-Schmidt vectors save.  A block's slice has
  // at most ceil(n / grid) elements plus the rows of the partial items at
  // both ends of its range.  r and w of the owned rows: an eighth.
  const size_t n = (size_t)sites * nc;
  const int gb = std::max(1, grid);
  const int ebound = (int)((n + gb - 1) / gb) + (int)((7LL * sites + gb - 1) / gb) + 2 * kMaxRows;
  const bool wsmem = (size_t)m * ebound * sizeof(float2) <= budget / 16;
  const bool esmem = 2 * (size_t)ebound * sizeof(float2) <= budget / 8;
  const size_t wbytes = (wsmem ? (size_t)m * ebound * sizeof(float2) : 0) + (esmem ? 2 * (size_t)ebound * sizeof(float2) : 0);
  int gsites = 4;
  for (int pass = 0; pass < 3; pass++) {
    const size_t other = fixed + wbytes + per_site * (size_t)gsites;
    p.stage_bytes = budget > other ? (int)(((budget - other) / stages) / 16 * 16) : 0;
    plan_items(p, sites, nc, nd, store);
    if (p.gmax <= gsites) break;
    gsites = p.gmax;
  }
  p.grid = std::min(grid, std::min(p.NA, p.NB));
  p.smem = (size_t)stages * p.stage_bytes + fixed + wbytes + per_site * (size_t)std::max(gsites, p.gmax);
  p.gmax = std::max(gsites, p.gmax);
  p.wsm_ld = wsmem ? ebound : 0;
  p.esm = esmem ? ebound : 0;
  if ((wsmem || esmem) && p.emax > ebound) raise(MG_ERR_STATE, "streamed coarse GCR: slice larger than planned");
  return p;
}

// 16 warps where their 32 stages hold items of two rows or more (Nc = 48 with a
// few sites per block), 8 otherwise: 16 halve the serial chain of a warp, two to
// three items per phase at 16^3x32.
Plan make_plan(const LevelGeom& G, const CoarseOp& C, int grid, int m) {
  const Plan p = plan_warps(G, C, grid, m, 16);
  return p.rowsA >= 2 ? p : plan_warps(G, C, grid, m, 8);
}

template <int W, int R>
const void* kernel_st(int store, bool eo) {
  return !eo                  ? (const void*)k_coarse_gcr_stream<kStF32, W, R, false>
         : store == STORE_F16  ? (const void*)k_coarse_gcr_stream<kStF16, W, R, true>
         : store == STORE_BF16 ? (const void*)k_coarse_gcr_stream<kStBF16, W, R, true>
                               : (const void*)k_coarse_gcr_stream<kStF32, W, R, true>;
}
const void* kernel_for(int store, bool eo, const Plan& p) {
  if (p.warps == 16)
    return p.rowsA == 8   ? kernel_st<16, 8>(store, eo)
           : p.rowsA == 4 ? kernel_st<16, 4>(store, eo)
                          : kernel_st<16, 2>(store, eo);
  return p.rowsA >= 2 ? kernel_st<8, 2>(store, eo) : kernel_st<8, 1>(store, eo);
}

int sm_count() {
  int dev = 0, sms = 0;
  MG_CUDA(cudaGetDevice(&dev));
  MG_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  return sms;
}

}  // namespace

// A stage holds a row of links, and the block fits with its static shared memory
// (below 512 bytes).  A smaller grid has more sites to gather per block and a shorter
// restart may place Krylov vectors in shared memory, so every (grid, m) is asked.
static bool plan_ok(const Plan& p) {
  return p.rowsA >= 1 && p.rowsB >= 1 && p.grid >= 1 && p.smem + 512 <= (size_t)p.optin;
}

std::vector<int> coarse_gcr_stream_grids(const LevelGeom& G, const CoarseOp& C, int m) {
  std::vector<int> out;
  if (C.nc % 2 || !C.A.get()) return out;
  const Plan p = make_plan(G, C, sm_count(), kMaxRestart);
  if (!plan_ok(p) || (m != kMaxRestart && !plan_ok(make_plan(G, C, p.grid, m)))) return out;
  out.push_back(p.grid);
  // the largest grid that splits both item lists evenly (no block waits at a
  // barrier for a neighbour with one more item)
  for (int g = p.grid - 1; g >= p.grid / 2 && g >= 1; g--)
    if (p.NA % g == 0 && p.NB % g == 0) {
      if (plan_ok(make_plan(G, C, g, m))) out.push_back(g);
      break;
    }
  return out;
}

void coarse_gcr_stream_solve(const LevelGeom& G, const CoarseOp& C, CoarseGCRBuffers& B, int m, int maxit,
                             double tol_rel, const float* b, float* x, long long* d_iters, int* flags, cudaStream_t s,
                             int grid) {
  if (m > kMaxRestart) raise(MG_ERR_ARG, "coarse restart too long for the persistent solver");
  if (C.nc % 2 || !C.A.get()) raise(MG_ERR_STATE, "streamed coarse solve not applicable to this level");
  const Plan p = make_plan(G, C, grid, m);
  if (!plan_ok(p)) raise(MG_ERR_STATE, "streamed coarse solve not applicable on this grid");
  const int sms = sm_count();
  int per = 0;
  const void* kern = kernel_for(C.store, G.eo, p);
  MG_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem));
  MG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, 32 * p.warps, p.smem));
  if (per < 1 || p.grid > per * sms) raise(MG_ERR_CUDA, "streamed coarse GCR cannot be resident");
  const size_t n = (size_t)(G.eo ? G.half : G.nsites) * C.nc;
  B.grow(B.st_part, sizeof(float2) * (size_t)kNR * p.grid);
  B.grow(B.st_sync, 256);
  if (B.W.bytes() < sizeof(float2) * n * m || B.Z.bytes() < sizeof(float2) * n * m)
    raise(MG_ERR_STATE, "coarse GCR buffers too small for this restart length");
  if (G.eo) {
    B.grow(B.st_to, sizeof(float2) * 2 * n);
    coarse_site_mul(G, C, true, G.half, G.nsites, B.st_to.as<float>(), b, s);     // t_o = X_o^{-1} b_o
  }
  MG_CUDA(cudaMemsetAsync(B.st_sync.get(), 0, 256, s));
  SArgs a;
  std::memset(&a, 0, sizeof(a));
  a.nc = C.nc;
  a.half = G.eo ? G.half : G.nsites;
  a.m = m;
  a.maxit = maxit;
  a.rowsA = p.rowsA;
  a.rowsB = p.rowsB;
  a.ipsA = p.ipsA;
  a.ipsB = p.ipsB;
  a.NA = G.eo ? p.NA : 0;
  a.NB = p.NB;
  a.eszB = !G.eo || C.store == STORE_F32 ? 8 : 4;
  a.stage_bytes = p.stage_bytes;
  a.gmax = p.gmax;
  a.wsm_ld = p.wsm_ld;
  a.esm = p.esm;
  a.tol_rel = tol_rel;
  a.nbr = G.d_nbr.as<int>();
  a.Y = static_cast<const unsigned char*>(G.eo ? C.Y.get() : C.A.get());
  a.Ys = C.Yscale.as<float>();
  a.Af = static_cast<const unsigned char*>(C.A.get());
  a.b = reinterpret_cast<const float2*>(b);
  a.to = B.st_to.as<float2>();
  a.x = reinterpret_cast<float2*>(x);
  a.y = G.eo ? B.y.as<float2>() : a.x;
  a.r = B.r.as<float2>();
  a.br = B.br.as<float2>();
  a.tB = B.tB.as<float2>();
  a.w = B.tA.as<float2>();
  a.W = B.W.as<float2>();
  a.Z = B.Z.as<float2>();
  a.partials = B.st_part.as<float2>();
  a.iters = d_iters;
  a.flags = flags;
  a.bar = B.st_sync.as<unsigned>();
  a.abort = reinterpret_cast<int*>(B.st_sync.as<unsigned char>() + 128);
  void* params[] = {&a};
  MG_CUDA(cudaLaunchCooperativeKernel(kern, dim3(p.grid), dim3(32 * p.warps), params, p.smem, s));
  MG_LAUNCH();
  if (G.eo) coarse_site_mul(G, C, true, 0, G.half, x, B.y.as<float>(), s);   // x_e = X_e^{-1} y_e; the kernel wrote x_o
}

}  // namespace mg
