// Coarse-level kernels of the adaptive multigrid (sm_103a).
//
//  * restriction R = P^dag and prolongation P with the chirality split of
//    the null vectors (section "Red-black preconditioning": P is built from
//    the low modes of D_p, split into the two chiralities inside each block;
//    R = P^dag gamma_5 gives the same coarse correction as R = P^dag for a
//    chirality-split P, so R = P^dag is applied)
//  * Galerkin coarse links D_hat = R D_p P ("Red-black preconditioning"):
//    one P column at a time, the eight directional hops of M^{-1} p are
//    projected onto the receiving block's P, hops across a block face into
//    Y_d and all others into X
//  * the coarse stencil D_hat v = X v + sum_d Y_d v(. + d) with the same
//    epilogues as the fine dslash, which give the coarse even-odd operators
//    (the coarse system is solved by its reduced even-odd form)
//  * FP64 batched Gauss-Jordan for X^{-1}
//  * block Gram-Schmidt (float-pair vectors and sums) and coarse-vector packing
//
// Coarse operators look like a staggered operator with Nc = 2 Nv colours
// ("Implementation"); a CTA owns one coarse site, its warps own rows of the
// 2Nv x 8*2Nv link block, and the neighbour vectors are staged in shared
// memory so each link row is read once, coalesced.
#include <algorithm>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "async_copy.cuh"
#include "coarse.h"
#include "coarse_dev.cuh"
#include "dfloat.cuh"
#include "philox.cuh"

namespace mg {

namespace {
constexpr int kBS = 256;

__device__ __forceinline__ cx<float> fget(const FineAccess& fa, const float* base, int idx, int c) {
  if (fa.wilson) {
    const int par = idx >= fa.Vh;
    const int cb = idx - par * fa.Vh;
    return SpinorIO<float>::get(base + (size_t)par * 24 * fa.Vh, fa.Vh, cb, c);
  }
  const float2 v = reinterpret_cast<const float2*>(base)[(size_t)idx * fa.ndof + c];
  return mkc(v.x, v.y);
}

__device__ __forceinline__ void fput(const FineAccess& fa, float* base, int idx, int c, cx<float> z) {
  if (fa.wilson) {
    const int par = idx >= fa.Vh;
    const int cb = idx - par * fa.Vh;
    SpinorIO<float>::put(base + (size_t)par * 24 * fa.Vh, fa.Vh, cb, c, z);
    return;
  }
  reinterpret_cast<float2*>(base)[(size_t)idx * fa.ndof + c] = make_float2(z.re, z.im);
}

// element e of a stored complex array in format ST
template <int ST>
__device__ __forceinline__ cx<float> sget(const void* p, size_t e) {
  if (ST == STORE_F32) {
    const float2 v = reinterpret_cast<const float2*>(p)[e];
    return mkc(v.x, v.y);
  } else if (ST == STORE_F16) {
    const float2 v = __half22float2(reinterpret_cast<const __half2*>(p)[e]);
    return mkc(v.x, v.y);
  } else {
    const float2 v = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(p)[e]);
    return mkc(v.x, v.y);
  }
}

template <int ST>
__device__ __forceinline__ void sput(void* p, size_t e, cx<float> z) {
  if (ST == STORE_F32) {
    reinterpret_cast<float2*>(p)[e] = make_float2(z.re, z.im);
  } else if (ST == STORE_F16) {
    reinterpret_cast<__half2*>(p)[e] = __floats2half2_rn(z.re, z.im);
  } else {
    reinterpret_cast<__nv_bfloat162*>(p)[e] = __floats2bfloat162_rn(z.re, z.im);
  }
}

struct TArgs {
  int nv, ndof, nb, fine_half, nbe;
  int b[4], cd[4];
  FineAccess fa;
  const int* blockmap;
  const int* evenlist;
  const void* P;
  const float* Ps;
  int* flags;
};

TArgs targs(const TransferOp& T) {
  TArgs a;
  a.nv = T.nv;
  a.ndof = T.fine_ndof;
  a.nb = T.nb;
  a.fine_half = T.fine_half;
  for (int m = 0; m < 4; m++) {
    a.b[m] = T.block[m];
    a.cd[m] = T.cdims[m];
  }
  a.fa = T.fa;
  a.nbe = T.nbe;
  a.blockmap = T.blockmap.as<int>();
  a.evenlist = T.evenlist.as<int>();
  a.P = T.P.get();
  a.Ps = T.Pscale.as<float>();
  a.flags = T.flags;
  return a;
}
}  // namespace

// --------------------------------------------------------------------------- restriction
// One CTA per coarse site and chirality.  Warp w takes the block's fine sites w,
// w+8, ...; lane k (and k+32 when Nv > 32) accumulates conj(P[i][c][k]) v[i][c].
// The site's components are read once by lanes 0..hd-1 and broadcast with
// shuffles; P rows are read coalesced, twelve in flight at a time: a coarse
// level has few blocks (32 of 2^4 sites here), so the time is a warp's chain of
// trips to L2 (both chiralities in one CTA with four rows in flight: 30 us,
// 15 us here, at Nc = 48).  Per-warp sums are combined in FP64 at the end.
template <int ST>
__global__ void __launch_bounds__(256) k_restrict(TArgs a, float* __restrict__ out, const float* __restrict__ v,
                                                  int even_only, int nrhs, size_t vstride, size_t cstride) {
  extern __shared__ float2 sacc[];  // [nwarps][nv]
  // one CTA per (coarse site, rhs), rhs fastest: the CTAs of a site share its P rows in L2
  const int cc = blockIdx.x / nrhs, rq = blockIdx.x % nrhs, ch = blockIdx.y;
  v += rq * vstride;
  out += rq * cstride;
  const int nv = a.nv, hd = a.ndof / 2;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  float acc[2][2] = {};  // [k-half][re, im]
  for (int i = w; i < a.nb; i += nw) {
    const int idx = a.blockmap[cc * a.nb + i];
    if (even_only && idx >= a.fine_half) continue;
    const cx<float> x = lane < hd ? fget(a.fa, v, idx, ch * hd + lane) : mkc(0.f, 0.f);
    const size_t base = (size_t)(cc * a.nb + i) * a.ndof + ch * hd;
#pragma unroll 12
    for (int c = 0; c < hd; c++) {
      const float xr = __shfl_sync(0xffffffffu, x.re, c);
      const float xi = __shfl_sync(0xffffffffu, x.im, c);
#pragma unroll
      for (int h = 0; h < 2; h++) {
        const int k = lane + 32 * h;
        if (k < nv) {
          const cx<float> p = sget<ST>(a.P, (base + c) * nv + k);
          acc[h][0] += p.re * xr + p.im * xi;
          acc[h][1] += p.re * xi - p.im * xr;
        }
      }
    }
  }
#pragma unroll
  for (int h = 0; h < 2; h++) {
    const int k = lane + 32 * h;
    if (k < nv) sacc[(size_t)w * nv + k] = make_float2(acc[h][0], acc[h][1]);
  }
  __syncthreads();
  const float sc = a.Ps[cc * 2 + ch];
  for (int t = threadIdx.x; t < nv; t += blockDim.x) {
    double re = 0, im = 0;
    for (int q = 0; q < nw; q++) {
      re += sacc[(size_t)q * nv + t].x;
      im += sacc[(size_t)q * nv + t].y;
    }
    reinterpret_cast<float2*>(out)[(size_t)cc * 2 * nv + ch * nv + t] = make_float2((float)(sc * re), (float)(sc * im));
  }
}

// Fine-level (Wilson) transfers.  One CTA per (coarse site, chirality, group
// of NR right-hand sides) walks the block's selected fine sites (all, or the
// even ones from the block's list) in tiles of kFTile sites through a
// kFStages-deep shared-memory pipeline.  A producer warp fills a stage --
// per site its P rows of the chirality, 6 Nv contiguous elements, with one
// bulk asynchronous copy each, and for the restriction the chirality's three
// float4 chunks of each right-hand side with 16-byte cp.async copies spread
// over its lanes (many tiny bulk copies would queue on the copy engine) --
// completed on the stage's "full" mbarrier; the consumer warps compute from
// the stage and release it on its "empty" mbarrier.  The bytes in flight per SM are set by the shared-memory budget
// (2-3 stages of each resident CTA), not by registers.  Every wait is bounded;
// a wait that runs out raises FLAG_TIMEOUT and the kernel carries on without
// it (every address stays in bounds), so the launch always ends.
constexpr int kFTile = 8;
constexpr int kFStages = 3;
constexpr int kFineMaxSites = 512;   // selected fine sites per block (indices kept in shared memory)

template <int ST>
__host__ __device__ constexpr int fine_esz() {
  return ST == STORE_F32 ? 8 : 4;
}

__host__ __device__ constexpr size_t align16(size_t x) { return (x + 15) & ~(size_t)15; }

bool fine_transfer_ok(const TransferOp& T, bool even_only, const void* fine, size_t fstride, const void* coarse,
                      size_t cstride) {
  return T.fa.wilson && T.nv <= 32 && T.nv % 2 == 0 && T.nb <= kFineMaxSites && (!even_only || T.nbe > 0) &&
         reinterpret_cast<uintptr_t>(fine) % 16 == 0 && reinterpret_cast<uintptr_t>(coarse) % 16 == 0 &&
         fstride % 4 == 0 && cstride % 4 == 0;
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

// an arrival on bar once all of the calling thread's earlier cp.async copies
// have landed (the barrier's expected count includes this arrival)
__device__ __forceinline__ void cp_async_arrive(uint64_t* bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void consumer_sync(int nthreads) {
  asm volatile("bar.sync 1, %0;" ::"r"(nthreads) : "memory");
}

// Restriction.  Consumer warp w takes the tile's sites w, w + 4; lane k < Nv
// accumulates conj(P[site][d][k]) x[site][d] (P from consecutive addresses, x
// as a broadcast).  The four warp sums are added in a fixed order.
constexpr int kRCons = 4;

template <int ST, int NR>
struct RestrictSmem {
  static constexpr int esz = fine_esz<ST>();
  int rowb, xoff, stb;
  size_t sacc, stage0, idx, total;
  __host__ __device__ RestrictSmem(int nv, int nsel) {
    rowb = 6 * nv * esz;
    xoff = kFTile * rowb;
    stb = xoff + kFTile * NR * 48;
    sacc = align16(sizeof(uint64_t) * 2 * kFStages);
    stage0 = align16(sacc + sizeof(float2) * kRCons * NR * 32);
    idx = stage0 + (size_t)kFStages * stb;
    total = idx + sizeof(int) * 2 * nsel;
  }
};

template <int ST, int NR>
__global__ void __launch_bounds__((kRCons + 1) * 32) k_restrict_fine(TArgs a, float* __restrict__ out,
                                                                     const float* __restrict__ v, int even_only,
                                                                     int nrhs, size_t vstride, size_t cstride) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int esz = fine_esz<ST>();
  const int nv = a.nv, Vh = a.fa.Vh;
  const int nsel = even_only ? a.nbe : a.nb;
  const RestrictSmem<ST, NR> L(nv, nsel);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem_raw);
  uint64_t* empty = full + kFStages;
  float2* sacc = reinterpret_cast<float2*>(smem_raw + L.sacc);   // [kRCons][NR][32]
  unsigned char* stage0 = smem_raw + L.stage0;
  int* si = reinterpret_cast<int*>(smem_raw + L.idx);            // [nsel] block-local index
  int* sx = si + nsel;                                           // [nsel] storage index
  const int nrg = (nrhs + NR - 1) / NR;
  const int cc = blockIdx.x / (2 * nrg), rem = blockIdx.x % (2 * nrg);
  const int ch = rem / nrg, r0 = (rem % nrg) * NR;
  const int nr = min(NR, nrhs - r0);
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (tid == 0) {
    for (int st = 0; st < kFStages; st++) {
      mbar_init(&full[st], 1 + 32);   // lane 0's arrival + every producer lane's cp.async arrival
      mbar_init(&empty[st], kRCons);
    }
    mbar_fence_init();
  }
  for (int t = tid; t < nsel; t += blockDim.x) {
    const int i = even_only ? a.evenlist[cc * a.nbe + t] : t;
    si[t] = i;
    sx[t] = a.blockmap[cc * a.nb + i];
  }
  __syncthreads();
  const int ntile = (nsel + kFTile - 1) / kFTile;
  bool ok = true;
  if (w == kRCons) {   // producer
    const unsigned char* Pb = static_cast<const unsigned char*>(a.P);
    for (int T = 0; T < ntile; T++) {
      const int st = T % kFStages, use = T / kFStages;
      if (use > 0) ok &= mbar_wait(&empty[st], (unsigned)((use - 1) & 1));
      const int s0 = T * kFTile, ns = min(kFTile, nsel - s0);
      unsigned char* sp = stage0 + (size_t)st * L.stb;
      if (lane == 0) mbar_expect_tx(&full[st], (unsigned)(ns * L.rowb));
      __syncwarp();
      if (lane < ns)
        bulk_copy_g2s(sp + lane * L.rowb, Pb + (((size_t)(cc * a.nb + si[s0 + lane]) * 12 + 6 * ch) * nv) * esz,
                      (unsigned)L.rowb, &full[st]);
      for (int u = lane; u < ns * nr * 3; u += 32) {
        const int s = u / (nr * 3), rq = u - s * nr * 3, r = rq / 3, q = rq - r * 3;
        const int idx = sx[s0 + s], par = idx >= Vh, cb = idx - par * Vh;
        cp_async16(sp + L.xoff + ((s * NR + r) * 3 + q) * 16,
                   reinterpret_cast<const float4*>(v + (size_t)(r0 + r) * vstride + (size_t)par * 24 * Vh) +
                       (size_t)(3 * ch + q) * Vh + cb);
      }
      cp_async_arrive(&full[st]);
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[st]);
    }
  } else {   // consumers
    float acc[NR][2];
#pragma unroll
    for (int r = 0; r < NR; r++) acc[r][0] = acc[r][1] = 0.f;
    for (int T = 0; T < ntile; T++) {
      const int st = T % kFStages, use = T / kFStages;
      ok &= mbar_wait(&full[st], (unsigned)(use & 1));
      const unsigned char* sp = stage0 + (size_t)st * L.stb;
      const float4* xs = reinterpret_cast<const float4*>(sp + L.xoff);
      const int ns = min(kFTile, nsel - T * kFTile);
      if (lane < nv) {
        for (int s = w; s < ns; s += kRCons) {
          const void* prow = sp + s * L.rowb;
#pragma unroll
          for (int d = 0; d < 6; d++) {
            const cx<float> p = sget<ST>(prow, (size_t)d * nv + lane);
#pragma unroll
            for (int r = 0; r < NR; r++) {
              if (r < nr) {
                const float4 c4 = xs[(s * NR + r) * 3 + (d >> 1)];
                const float xr = (d & 1) ? c4.z : c4.x, xi = (d & 1) ? c4.w : c4.y;
                acc[r][0] = fmaf(p.re, xr, fmaf(p.im, xi, acc[r][0]));
                acc[r][1] = fmaf(p.re, xi, fmaf(-p.im, xr, acc[r][1]));
              }
            }
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[st]);
    }
#pragma unroll
    for (int r = 0; r < NR; r++) sacc[(w * NR + r) * 32 + lane] = make_float2(acc[r][0], acc[r][1]);
    consumer_sync(kRCons * 32);
    const float sc = a.Ps[cc * 2 + ch];
    for (int t = tid; t < nr * nv; t += kRCons * 32) {
      const int r = t / nv, k = t - r * nv;
      float re = 0.f, im = 0.f;
#pragma unroll
      for (int q = 0; q < kRCons; q++) {
        re += sacc[(q * NR + r) * 32 + k].x;
        im += sacc[(q * NR + r) * 32 + k].y;
      }
      reinterpret_cast<float2*>(out + (size_t)(r0 + r) * cstride)[(size_t)cc * 2 * nv + ch * nv + k] =
          make_float2(sc * re, sc * im);
    }
  }
  if (!ok && a.flags) atomicExch(&a.flags[FLAG_TIMEOUT], 1);
}

template <int ST, int NR>
void launch_restrict_fine(const TArgs& a, int ncoarse, int nrhs, float* out, const float* v, bool even_only,
                          size_t vstride, size_t cstride, cudaStream_t s) {
  const unsigned grid = (unsigned)((size_t)ncoarse * 2 * ((nrhs + NR - 1) / NR));
  const RestrictSmem<ST, NR> L(a.nv, even_only ? a.nbe : a.nb);
  MG_CUDA(cudaFuncSetAttribute(k_restrict_fine<ST, NR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L.total));
  k_restrict_fine<ST, NR><<<grid, (kRCons + 1) * 32, L.total, s>>>(a, out, v, even_only, nrhs, vstride, cstride);
  MG_LAUNCH();
}

template <int ST>
void restrict_fine(const TArgs& a, int ncoarse, int nrhs, float* out, const float* v, bool even_only,
                   size_t vstride, size_t cstride, cudaStream_t s) {
  if (nrhs >= 4)
    launch_restrict_fine<ST, 4>(a, ncoarse, nrhs, out, v, even_only, vstride, cstride, s);
  else if (nrhs >= 2)
    launch_restrict_fine<ST, 2>(a, ncoarse, nrhs, out, v, even_only, vstride, cstride, s);
  else
    launch_restrict_fine<ST, 1>(a, ncoarse, nrhs, out, v, even_only, vstride, cstride, s);
}

void restrict_vec_multi(const TransferOp& T, int nrhs, float* out_c, size_t cstride, const float* v, size_t vstride,
                        bool even_only, cudaStream_t s) {
  TArgs a = targs(T);
  if (fine_transfer_ok(T, even_only, v, vstride, out_c, cstride)) {
    switch (T.store) {
      case STORE_F32: restrict_fine<STORE_F32>(a, T.ncoarse, nrhs, out_c, v, even_only, vstride, cstride, s); break;
      case STORE_F16: restrict_fine<STORE_F16>(a, T.ncoarse, nrhs, out_c, v, even_only, vstride, cstride, s); break;
      default: restrict_fine<STORE_BF16>(a, T.ncoarse, nrhs, out_c, v, even_only, vstride, cstride, s); break;
    }
    return;
  }
  const size_t sm = sizeof(float2) * (kBS / 32) * (size_t)T.nv;
  const dim3 grid((unsigned)((size_t)T.ncoarse * nrhs), 2);
  switch (T.store) {
    case STORE_F32: k_restrict<STORE_F32><<<grid, kBS, sm, s>>>(a, out_c, v, even_only, nrhs, vstride, cstride); break;
    case STORE_F16: k_restrict<STORE_F16><<<grid, kBS, sm, s>>>(a, out_c, v, even_only, nrhs, vstride, cstride); break;
    default: k_restrict<STORE_BF16><<<grid, kBS, sm, s>>>(a, out_c, v, even_only, nrhs, vstride, cstride); break;
  }
  MG_LAUNCH();
}

void restrict_vec(const TransferOp& T, float* out_c, const float* v, bool even_only, cudaStream_t s) {
  restrict_vec_multi(T, 1, out_c, 0, v, 0, even_only, s);
}

// --------------------------------------------------------------------------- prolongation
template <int ST>
__global__ void k_prolong(TArgs a, float* __restrict__ v, const float* __restrict__ in_c, int even_only, int nrhs,
                          size_t vstride, size_t cstride) {
  extern __shared__ float2 svc[];  // [2 nv]
  const int cc = blockIdx.x / nrhs, rq = blockIdx.x % nrhs;   // (coarse site, rhs), rhs fastest
  v += rq * vstride;
  in_c += rq * cstride;
  const int nv = a.nv, hd = a.ndof / 2;
  for (int t = threadIdx.x; t < 2 * nv; t += blockDim.x)
    svc[t] = reinterpret_cast<const float2*>(in_c)[(size_t)cc * 2 * nv + t];
  __syncthreads();
  const float s0 = a.Ps[cc * 2], s1 = a.Ps[cc * 2 + 1];
  for (int t = threadIdx.x; t < a.nb * a.ndof; t += blockDim.x) {
    const int i = t / a.ndof, c = t % a.ndof;
    const int idx = a.blockmap[cc * a.nb + i];
    if (even_only && idx >= a.fine_half) continue;
    const int ch = c >= hd;
    const float2* vc = svc + ch * nv;
    const size_t base = ((size_t)(cc * a.nb + i) * a.ndof + c) * nv;
    float re = 0.f, im = 0.f;
    for (int k = 0; k < nv; k++) {
      const cx<float> p = sget<ST>(a.P, base + k);
      re += p.re * vc[k].x - p.im * vc[k].y;
      im += p.re * vc[k].y + p.im * vc[k].x;
    }
    const float sc = ch ? s1 : s0;
    fput(a.fa, v, idx, c, mkc(sc * re, sc * im));
  }
}

// Prolongation onto the fine (Wilson) level, with the pipeline of the
// restriction (one CTA per (coarse site, chirality, group of NR right-hand
// sides)); the producer also copies the coarse vectors of the chirality once.
// Consumer warp w forms the float4 chunk 3 ch + w (spin-colour components
// 6 ch + 2w, +1) of the tile's sites: lane = site (lane & 7) + 8 g, the four
// g lanes of a site taking its NR right-hand sides, each split over 4 / NR
// lanes that share the Nv/2 pairs of null vectors and add their sums with
// shuffles; one lane per (site, right-hand side) stores the chunk with one
// 16-byte store.  A staged site occupies an odd
// number of 16-byte units, so the eight sites of a quarter-warp read
// different banks; the coarse vector is read as a broadcast.
constexpr int kPCons = 3;

template <int ST, int NR>
struct ProlongSmem {
  static constexpr int esz = fine_esz<ST>();
  int rowb, pitch, stb;
  size_t svc, stage0, idx, total;
  __host__ __device__ ProlongSmem(int nv, int nsel) {
    rowb = 6 * nv * esz;
    pitch = 16 * ((rowb / 16) | 1);
    stb = kFTile * pitch;
    svc = align16(sizeof(uint64_t) * (2 * kFStages + 1));
    stage0 = align16(svc + sizeof(float2) * NR * nv);
    idx = stage0 + (size_t)kFStages * stb;
    total = idx + sizeof(int) * 2 * nsel;
  }
};

template <int ST, int NR>
__global__ void __launch_bounds__((kPCons + 1) * 32) k_prolong_fine(TArgs a, float* __restrict__ v,
                                                                    const float* __restrict__ in_c, int even_only,
                                                                    int nrhs, size_t vstride, size_t cstride) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int esz = fine_esz<ST>();
  const int nv = a.nv, Vh = a.fa.Vh;
  const int nsel = even_only ? a.nbe : a.nb;
  const ProlongSmem<ST, NR> L(nv, nsel);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem_raw);
  uint64_t* empty = full + kFStages;
  uint64_t* cbar = empty + kFStages;
  const float2* svc = reinterpret_cast<const float2*>(smem_raw + L.svc);   // [NR][nv]
  unsigned char* stage0 = smem_raw + L.stage0;
  int* si = reinterpret_cast<int*>(smem_raw + L.idx);
  int* sx = si + nsel;
  const int nrg = (nrhs + NR - 1) / NR;
  const int cc = blockIdx.x / (2 * nrg), rem = blockIdx.x % (2 * nrg);
  const int ch = rem / nrg, r0 = (rem % nrg) * NR;
  const int nr = min(NR, nrhs - r0);
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (tid == 0) {
    for (int st = 0; st < kFStages; st++) {
      mbar_init(&full[st], 1);
      mbar_init(&empty[st], kPCons);
    }
    mbar_init(cbar, 1);
    mbar_fence_init();
  }
  for (int t = tid; t < nsel; t += blockDim.x) {
    const int i = even_only ? a.evenlist[cc * a.nbe + t] : t;
    si[t] = i;
    sx[t] = a.blockmap[cc * a.nb + i];
  }
  __syncthreads();
  const int ntile = (nsel + kFTile - 1) / kFTile;
  bool ok = true;
  if (w == kPCons) {   // producer
    if (lane == 0) mbar_expect_tx(cbar, (unsigned)(nr * nv * 8));
    __syncwarp();
    if (lane < nr)
      bulk_copy_g2s(smem_raw + L.svc + (size_t)lane * nv * 8,
                    in_c + (size_t)(r0 + lane) * cstride + ((size_t)cc * 2 * nv + ch * nv) * 2, (unsigned)(nv * 8),
                    cbar);
    __syncwarp();
    if (lane == 0) mbar_arrive(cbar);
    const unsigned char* Pb = static_cast<const unsigned char*>(a.P);
    for (int T = 0; T < ntile; T++) {
      const int st = T % kFStages, use = T / kFStages;
      if (use > 0) ok &= mbar_wait(&empty[st], (unsigned)((use - 1) & 1));
      const int s0 = T * kFTile, ns = min(kFTile, nsel - s0);
      if (lane == 0) mbar_expect_tx(&full[st], (unsigned)(ns * L.rowb));
      __syncwarp();
      if (lane < ns)
        bulk_copy_g2s(stage0 + (size_t)st * L.stb + lane * L.pitch,
                      Pb + (((size_t)(cc * a.nb + si[s0 + lane]) * 12 + 6 * ch) * nv) * esz, (unsigned)L.rowb,
                      &full[st]);
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[st]);
    }
  } else {   // consumers
    ok &= mbar_wait(cbar, 0u);
    constexpr int KQ = 4 / NR;   // lanes sharing the pairs of one (site, right-hand side)
    const int s = lane & 7, g = lane >> 3, rq = g / KQ, kq = g % KQ;
    const int npair = nv / 2;
    const float4* c2p = reinterpret_cast<const float4*>(svc + rq * nv);
    for (int T = 0; T < ntile; T++) {
      const int st = T % kFStages, use = T / kFStages;
      ok &= mbar_wait(&full[st], (unsigned)(use & 1));
      const int s0 = T * kFTile, ns = min(kFTile, nsel - s0);
      const unsigned char* row0 = stage0 + (size_t)st * L.stb + s * L.pitch + 2 * w * nv * esz;
      const unsigned char* row1 = row0 + nv * esz;
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
      if (s < ns && rq < nr) {
        for (int kp = kq; kp < npair; kp += KQ) {
          float2 p0[2], p1[2];
          if (ST == STORE_F32) {
            const float4 u0 = reinterpret_cast<const float4*>(row0)[kp];
            const float4 u1 = reinterpret_cast<const float4*>(row1)[kp];
            p0[0] = make_float2(u0.x, u0.y);
            p0[1] = make_float2(u0.z, u0.w);
            p1[0] = make_float2(u1.x, u1.y);
            p1[1] = make_float2(u1.z, u1.w);
          } else {
            const uint2 u0 = reinterpret_cast<const uint2*>(row0)[kp];
            const uint2 u1 = reinterpret_cast<const uint2*>(row1)[kp];
            if (ST == STORE_F16) {
              p0[0] = __half22float2(*reinterpret_cast<const __half2*>(&u0.x));
              p0[1] = __half22float2(*reinterpret_cast<const __half2*>(&u0.y));
              p1[0] = __half22float2(*reinterpret_cast<const __half2*>(&u1.x));
              p1[1] = __half22float2(*reinterpret_cast<const __half2*>(&u1.y));
            } else {
              p0[0] = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u0.x));
              p0[1] = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u0.y));
              p1[0] = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u1.x));
              p1[1] = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u1.y));
            }
          }
          const float4 c2 = c2p[kp];
#pragma unroll
          for (int h = 0; h < 2; h++) {
            const float cr = h ? c2.z : c2.x, ci = h ? c2.w : c2.y;
            acc[0] = fmaf(p0[h].x, cr, fmaf(-p0[h].y, ci, acc[0]));
            acc[1] = fmaf(p0[h].x, ci, fmaf(p0[h].y, cr, acc[1]));
            acc[2] = fmaf(p1[h].x, cr, fmaf(-p1[h].y, ci, acc[2]));
            acc[3] = fmaf(p1[h].x, ci, fmaf(p1[h].y, cr, acc[3]));
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[st]);   // the stage is read; what follows uses registers
#pragma unroll
      for (int o = 8; o < 8 * KQ; o <<= 1)
#pragma unroll
        for (int e = 0; e < 4; e++) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], o);
      if (s < ns && rq < nr && kq == 0) {
        const float sc = a.Ps[cc * 2 + ch];
        const int idx = sx[s0 + s], par = idx >= Vh, cb = idx - par * Vh;
        reinterpret_cast<float4*>(v + (size_t)(r0 + rq) * vstride + (size_t)par * 24 * Vh)[(size_t)(3 * ch + w) * Vh +
                                                                                           cb] =
            make_float4(sc * acc[0], sc * acc[1], sc * acc[2], sc * acc[3]);
      }
    }
  }
  if (!ok && a.flags) atomicExch(&a.flags[FLAG_TIMEOUT], 1);
}

template <int ST, int NR>
void launch_prolong_fine(const TArgs& a, const TransferOp& T, int nrhs, float* v, const float* in_c, bool even_only,
                         size_t vstride, size_t cstride, cudaStream_t s) {
  const unsigned grid = (unsigned)((size_t)T.ncoarse * 2 * ((nrhs + NR - 1) / NR));
  const ProlongSmem<ST, NR> L(T.nv, even_only ? T.nbe : T.nb);
  MG_CUDA(cudaFuncSetAttribute(k_prolong_fine<ST, NR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L.total));
  k_prolong_fine<ST, NR><<<grid, (kPCons + 1) * 32, L.total, s>>>(a, v, in_c, even_only, nrhs, vstride, cstride);
  MG_LAUNCH();
}

template <int ST>
void prolong_fine(const TArgs& a, const TransferOp& T, int nrhs, float* v, const float* in_c, bool even_only,
                  size_t vstride, size_t cstride, cudaStream_t s) {
  if (nrhs >= 4)
    launch_prolong_fine<ST, 4>(a, T, nrhs, v, in_c, even_only, vstride, cstride, s);
  else if (nrhs >= 2)
    launch_prolong_fine<ST, 2>(a, T, nrhs, v, in_c, even_only, vstride, cstride, s);
  else
    launch_prolong_fine<ST, 1>(a, T, nrhs, v, in_c, even_only, vstride, cstride, s);
}

void prolong_vec_multi(const TransferOp& T, int nrhs, float* v, size_t vstride, const float* in_c, size_t cstride,
                       bool even_only, cudaStream_t s) {
  TArgs a = targs(T);
  if (fine_transfer_ok(T, even_only, v, vstride, in_c, cstride)) {
    switch (T.store) {
      case STORE_F32: prolong_fine<STORE_F32>(a, T, nrhs, v, in_c, even_only, vstride, cstride, s); break;
      case STORE_F16: prolong_fine<STORE_F16>(a, T, nrhs, v, in_c, even_only, vstride, cstride, s); break;
      default: prolong_fine<STORE_BF16>(a, T, nrhs, v, in_c, even_only, vstride, cstride, s); break;
    }
    return;
  }
  const size_t sm = sizeof(float2) * 2 * T.nv;
  const unsigned grid = (unsigned)((size_t)T.ncoarse * nrhs);
  switch (T.store) {
    case STORE_F32: k_prolong<STORE_F32><<<grid, kBS, sm, s>>>(a, v, in_c, even_only, nrhs, vstride, cstride); break;
    case STORE_F16: k_prolong<STORE_F16><<<grid, kBS, sm, s>>>(a, v, in_c, even_only, nrhs, vstride, cstride); break;
    default: k_prolong<STORE_BF16><<<grid, kBS, sm, s>>>(a, v, in_c, even_only, nrhs, vstride, cstride); break;
  }
  MG_LAUNCH();
}

void prolong_vec(const TransferOp& T, float* v, const float* in_c, bool even_only, cudaStream_t s) {
  prolong_vec_multi(T, 1, v, 0, in_c, 0, even_only, s);
}

// --------------------------------------------------------------------------- column extraction
// column0 + blockIdx.y of P (column = chirality * Nv + k) as a whole-lattice vector
template <int ST>
__global__ void k_extract_columns(TArgs a, float* p, size_t vstride, int column0) {
  const size_t total = (size_t)a.nb * a.ndof;
  const int cc = blockIdx.x;
  const int hd = a.ndof / 2;
  const int col = column0 + blockIdx.y, chir = col / a.nv, k = col % a.nv;
  p += blockIdx.y * vstride;
  for (size_t t = threadIdx.x; t < total; t += blockDim.x) {
    const int i = (int)(t / a.ndof), c = (int)(t % a.ndof);
    const int idx = a.blockmap[cc * a.nb + i];
    cx<float> z = mkc(0.f, 0.f);
    if ((c >= hd) == (chir == 1)) {
      z = sget<ST>(a.P, ((size_t)(cc * a.nb + i) * a.ndof + c) * a.nv + k);
      const float sc = a.Ps[cc * 2 + chir];
      z = mkc(sc * z.re, sc * z.im);
    }
    fput(a.fa, p, idx, c, z);
  }
}

void extract_columns(const TransferOp& T, float* p, size_t vstride, int column0, int ncol, cudaStream_t s) {
  TArgs a = targs(T);
  const dim3 grid(T.ncoarse, ncol);
  switch (T.store) {
    case STORE_F32: k_extract_columns<STORE_F32><<<grid, kBS, 0, s>>>(a, p, vstride, column0); break;
    case STORE_F16: k_extract_columns<STORE_F16><<<grid, kBS, 0, s>>>(a, p, vstride, column0); break;
    default: k_extract_columns<STORE_BF16><<<grid, kBS, 0, s>>>(a, p, vstride, column0); break;
  }
  MG_LAUNCH();
}

// --------------------------------------------------------------------------- Galerkin columns
// The columns' directional hops W_d of u = M^{-1} p projected on P^dag.  Hops
// that stay inside the block all end in X, so they are summed before the
// projection (together with the identity-slot vector): the interior sum is
// kept as an unevaluated float pair (about 48 bits), and only the hops that
// cross a block face are projected one by one.  Per site of a 4^4 block that
// is 1 + 2 projections instead of 9.  The inner products are bound by
// arithmetic: FP64 runs at 1/62 of the FP32 rate on GB300, so every product
// is accumulated in compensated FP32 (error-free product and sum, ten FP32
// operations, about 48 bits) and the per-thread sums are added in FP64.
// Measured on 16^3x32 (4^4 blocks, Nv = 24, 48 columns): 383 ms with nine
// FP64 projections per site, 15.2 ms now (24 launches of two columns), the
// hops and column extraction around them 2.2 ms.

// complex conj(p) w
__device__ __forceinline__ void dot2_cacc(float (&a)[4], cx<float> p, float wr, float wi) {
  dot2_acc(a[0], a[1], p.re, wr);
  dot2_acc(a[0], a[1], p.im, wi);
  dot2_acc(a[2], a[3], p.re, wi);
  dot2_acc(a[2], a[3], -p.im, wr);
}

// interior sums of a coarse-level column from its nine whole-lattice vectors
// (AoS vectors); one CTA per (block, column)
struct W8 {
  const float* p[8];
};
__device__ __forceinline__ void block_coords(const TArgs& a, int i, int l[4]) {
  l[0] = i % a.b[0];
  i /= a.b[0];
  l[1] = i % a.b[1];
  i /= a.b[1];
  l[2] = i % a.b[2];
  l[3] = i / a.b[2];
}
__global__ void k_interior_sum(TArgs a, W8 W, const float* slot, float* Sh, float* Sl, size_t vstride) {
  const int cc = blockIdx.x;
  const size_t o = blockIdx.y * vstride;
  for (int t = threadIdx.x; t < a.nb * a.ndof; t += blockDim.x) {
    const int i = t / a.ndof, c = t % a.ndof;
    const size_t e = o + 2 * ((size_t)a.blockmap[cc * a.nb + i] * a.ndof + c);
    int l[4];
    block_coords(a, i, l);
    float h[2] = {slot[e], slot[e + 1]}, lo[2] = {0.f, 0.f};
#pragma unroll
    for (int d = 0; d < 8; d++) {
      const int mu = d & 3;
      if (a.cd[mu] > 1 && (d < 4 ? l[mu] == a.b[mu] - 1 : l[mu] == 0)) continue;
      for (int q = 0; q < 2; q++) df_acc(h[q], lo[q], W.p[d][e + q]);
    }
    for (int q = 0; q < 2; q++) {
      Sh[e + q] = h[q];
      Sl[e + q] = lo[q];
    }
  }
}

void interior_sum(const TransferOp& T, const float* const W[8], const float* slot, float* Sh, float* Sl,
                  size_t vstride, int ncol, cudaStream_t s) {
  W8 w;
  for (int d = 0; d < 8; d++) w.p[d] = W[d];
  k_interior_sum<<<dim3(T.ncoarse, ncol), kBS, 0, s>>>(targs(T), w, slot, Sh, Sl, vstride);
  MG_LAUNCH();
}

// Rows of Y (face hops) and X (interior sum) of columns col0 + 2 blockIdx.y, + 1.
// CTA = (block, row chirality) x two columns x one part (0: the interior sum
// over all nb sites; 1, 2: the four forward / backward face hops, nb / b_mu
// sites each), so the three parts have the same work on a hypercubic block.
// Thread (k, g) takes null vector k and the sites g, g + G, ...: threads of a
// site read its P row contiguously and its vector as a broadcast, every P
// entry serves two columns, and a thread holds the sums of one hop only (eight
// registers), so occupancy hides the load latency.
template <int ST>
__global__ void __launch_bounds__(kBS) k_galerkin_project(TArgs a, W8 W, const float* Sh, const float* Sl,
                                                          size_t vstride, float2* __restrict__ Y,
                                                          float2* __restrict__ X, int col0) {
  __shared__ double sred[4 * kBS];   // [column 2][re, im][thread]
  const int cc = blockIdx.x >> 1, ch = blockIdx.x & 1;
  const int nv = a.nv, G = kBS / nv, nc = 2 * nv;
  const int k = threadIdx.x % nv, g = threadIdx.x / nv;
  const int hd = a.ndof / 2;
  const size_t o0 = (size_t)(2 * blockIdx.y) * vstride, o1 = o0 + vstride;
  const float sc = a.Ps[cc * 2 + ch];
  const int d0 = blockIdx.z == 2 ? 4 : 0, d1 = blockIdx.z == 0 ? 1 : d0 + 4;
  for (int d = d0; d < d1; d++) {
    const bool interior = blockIdx.z == 0;
    const int mu = d & 3;
    int below = 1;
    for (int m = 0; m < mu; m++) below *= a.b[m];
    const int at = d < 4 ? a.b[mu] - 1 : 0;
    const int cnt = interior ? a.nb : (a.cd[mu] > 1 ? a.nb / a.b[mu] : 0);
    const float* w0 = interior ? Sh : W.p[d];
    float acc[2][4] = {};
    if (g < G)
      for (int t = g; t < cnt; t += G) {
        const int i = interior ? t : t % below + below * at + (t / below) * below * a.b[mu];
        const int idx = a.blockmap[cc * a.nb + i];
        const size_t prow = ((size_t)(cc * a.nb + i) * a.ndof + ch * hd) * nv + k;
        auto entry = [&](int c) {
          const cx<float> p = sget<ST>(a.P, prow + (size_t)c * nv);
          return mkc(sc * p.re, sc * p.im);
        };
        const size_t e0 = 2 * ((size_t)idx * a.ndof + ch * hd);
        for (int c = 0; c < hd; c++) {
          const cx<float> p = entry(c);
#pragma unroll
          for (int q = 0; q < 2; q++) {
            const size_t e = (q ? o1 : o0) + e0 + 2 * c;
            const float2 x = *reinterpret_cast<const float2*>(w0 + e);
            dot2_cacc(acc[q], p, x.x, x.y);
            if (interior) {   // the low halves: first-order corrections
              const float2 y = *reinterpret_cast<const float2*>(Sl + e);
              acc[q][1] = fmaf(p.re, y.x, fmaf(p.im, y.y, acc[q][1]));
              acc[q][3] = fmaf(p.re, y.y, fmaf(-p.im, y.x, acc[q][3]));
            }
          }
        }
      }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 2; q++) {
      sred[(2 * q) * kBS + threadIdx.x] = g < G ? (double)acc[q][0] + (double)acc[q][1] : 0.0;
      sred[(2 * q + 1) * kBS + threadIdx.x] = g < G ? (double)acc[q][2] + (double)acc[q][3] : 0.0;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < 2 * nv; t += kBS) {
      const int q = t / nv, kk = t % nv;
      double re = 0, im = 0;
      for (int gg = 0; gg < G; gg++) {
        re += sred[(2 * q) * kBS + gg * nv + kk];
        im += sred[(2 * q + 1) * kBS + gg * nv + kk];
      }
      const size_t row = (size_t)cc * nc + ch * nv + kk;
      const int col = col0 + 2 * blockIdx.y + q;
      if (interior)
        X[row * nc + col] = make_float2((float)re, (float)im);
      else
        Y[(row * 8 + d) * nc + col] = make_float2((float)re, (float)im);
    }
  }
}


// The same from the fine level.  With each thread loading what it multiplies,
// warps waited for L2 two thirds of the time (issue slots 50 % used, 52
// registers, four CTAs per SM).  Here tiles of G sites -- their P rows of the
// chirality, contiguous, and the vectors of both columns -- are copied to shared
// memory three tiles deep (cp.async), the block map entry one tile further
// ahead: 631 -> 527 us per launch of two columns at 16^3x32.
constexpr int kGalStages = 3;
template <int ST>
__global__ void __launch_bounds__(kBS) k_galerkin_project_fine(TArgs a, W8 W, const float* Sh, const float* Sl,
                                                               size_t vstride, float2* __restrict__ Y,
                                                               float2* __restrict__ X, int col0) {
  extern __shared__ __align__(16) unsigned char gsm[];   // [stage]: [G][12] float4, [G][6 Nv] entries of P
  __shared__ double sred[4 * kBS];                       // [column 2][re, im][thread]
  constexpr int esz = ST == STORE_F32 ? 8 : 4, chunk = 2 * esz;   // 3 Nv chunks of P per site
  const int cc = blockIdx.x >> 1, ch = blockIdx.x & 1;
  const int nv = a.nv, G = kBS / nv, nc = 2 * nv;
  const int k = threadIdx.x % nv, g = threadIdx.x / nv;
  const int pbytes = 6 * nv * esz, stage_bytes = (G * (192 + pbytes) + 15) / 16 * 16;
  const size_t o0 = (size_t)(2 * blockIdx.y) * vstride;
  const float sc = a.Ps[cc * 2 + ch];
  const bool interior = blockIdx.z == 0;
  const int d0 = blockIdx.z == 2 ? 4 : 0, d1 = interior ? 1 : d0 + 4;
  auto count = [&](int d) { return interior ? a.nb : (a.cd[d & 3] > 1 ? a.nb / a.b[d & 3] : 0); };
  auto site_of = [&](int d, int t) {   // site t of the face that hop d crosses
    if (interior) return t;
    const int mu = d & 3;
    int below = 1;
    for (int m = 0; m < mu; m++) below *= a.b[m];
    return t % below + below * (d < 4 ? a.b[mu] - 1 : 0) + (t / below) * below * a.b[mu];
  };
  // the next tile to copy, and this group's site of it
  int pd = d0, pt = 0, pi = -1, pidx = 0;
  auto peek = [&]() {
    while (pd < d1 && pt * G >= count(pd)) {
      pd++;
      pt = 0;
    }
    pi = -1;
    if (g < G && pd < d1 && pt * G + g < count(pd)) {
      pi = site_of(pd, pt * G + g);
      pidx = a.blockmap[cc * a.nb + pi];
    }
  };
  auto copy = [&](int stage) {
    if (pi >= 0) {
      unsigned char* base = gsm + (size_t)stage * stage_bytes;
      const unsigned char* psrc = static_cast<const unsigned char*>(a.P) + ((size_t)(cc * a.nb + pi) * 12 + ch * 6) * nv * esz;
      unsigned char* pdst = base + G * 192 + g * pbytes;
#pragma unroll
      for (int j = 0; j < 3; j++) {
        const int o = (j * nv + k) * chunk;
        if (chunk == 16)
          cp_async16(pdst + o, psrc + o);
        else
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(pdst + o)), "l"(psrc + o) : "memory");
      }
      const int par = pidx >= a.fa.Vh, cb = pidx - par * a.fa.Vh;
      const size_t e0 = o0 + (size_t)par * 24 * a.fa.Vh + 4 * (size_t)cb;
      for (int q = k; q < (interior ? 12 : 6); q += nv) {   // (high, low half), column, component pair
        const float* v = q >= 6 ? Sl : interior ? Sh : W.p[pd];
        cp_async16(base + (g * 12 + q) * 16, v + e0 + (q / 3 & 1) * vstride + (size_t)(3 * ch + q % 3) * 4 * a.fa.Vh);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    pt++;
    peek();
  };
  peek();
  for (int st = 0; st < kGalStages - 1; st++) copy(st);
  int step = 0;
  for (int d = d0; d < d1; d++) {
    const int cnt = count(d);
    float acc[2][4] = {};
    for (int t0 = 0; t0 < cnt; t0 += G, step++) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kGalStages - 2) : "memory");
      __syncthreads();
      copy((step + kGalStages - 1) % kGalStages);   // the tile consumed before this barrier
      if (g < G && t0 + g < cnt) {
        const unsigned char* base = gsm + (size_t)(step % kGalStages) * stage_bytes;
        const float4* vec = reinterpret_cast<const float4*>(base) + g * 12;
        const unsigned char* prow = base + G * 192 + g * pbytes;
#pragma unroll
        for (int c = 0; c < 3; c++) {
          cx<float> p0 = sget<ST>(prow, (size_t)(2 * c) * nv + k), p1 = sget<ST>(prow, (size_t)(2 * c + 1) * nv + k);
          p0 = mkc(sc * p0.re, sc * p0.im);
          p1 = mkc(sc * p1.re, sc * p1.im);
#pragma unroll
          for (int q = 0; q < 2; q++) {
            const float4 x = vec[3 * q + c];
            dot2_cacc(acc[q], p0, x.x, x.y);
            dot2_cacc(acc[q], p1, x.z, x.w);
            if (interior) {   // the low halves: first-order corrections
              const float4 y = vec[6 + 3 * q + c];
              acc[q][1] = fmaf(p0.re, y.x, fmaf(p0.im, y.y, acc[q][1]));
              acc[q][3] = fmaf(p0.re, y.y, fmaf(-p0.im, y.x, acc[q][3]));
              acc[q][1] = fmaf(p1.re, y.z, fmaf(p1.im, y.w, acc[q][1]));
              acc[q][3] = fmaf(p1.re, y.w, fmaf(-p1.im, y.z, acc[q][3]));
            }
          }
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 2; q++) {
      sred[(2 * q) * kBS + threadIdx.x] = g < G ? (double)acc[q][0] + (double)acc[q][1] : 0.0;
      sred[(2 * q + 1) * kBS + threadIdx.x] = g < G ? (double)acc[q][2] + (double)acc[q][3] : 0.0;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < 2 * nv; t += kBS) {
      const int q = t / nv, kk = t % nv;
      double re = 0, im = 0;
      for (int gg = 0; gg < G; gg++) {
        re += sred[(2 * q) * kBS + gg * nv + kk];
        im += sred[(2 * q + 1) * kBS + gg * nv + kk];
      }
      const size_t row = (size_t)cc * nc + ch * nv + kk;
      const int col = col0 + 2 * blockIdx.y + q;
      if (interior)
        X[row * nc + col] = make_float2((float)re, (float)im);
      else
        Y[(row * 8 + d) * nc + col] = make_float2((float)re, (float)im);
    }
  }
}

void galerkin_project(const TransferOp& T, CoarseOp& C, const float* const W[8], const float* Sh, const float* Sl,
                      size_t vstride, int col0, int ncol, cudaStream_t s) {
  if (ncol % 2) raise(MG_ERR_ARG, "Galerkin columns are projected in pairs");
  const TArgs a = targs(T);
  W8 w;
  for (int d = 0; d < 8; d++) w.p[d] = W[d];
  const dim3 grid(T.ncoarse * 2, ncol / 2, 3);
  float2* Y = C.Y.as<float2>();
  float2* X = C.X.as<float2>();
  auto run = [&](auto st) {
    constexpr int ST = decltype(st)::value;
    if (T.fa.wilson) {
      const int sm = kGalStages * (((kBS / T.nv) * (192 + 6 * T.nv * (ST == STORE_F32 ? 8 : 4)) + 15) / 16 * 16);
      MG_CUDA(cudaFuncSetAttribute(k_galerkin_project_fine<ST>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm));
      k_galerkin_project_fine<ST><<<grid, kBS, sm, s>>>(a, w, Sh, Sl, vstride, Y, X, col0);
    } else {
      k_galerkin_project<ST><<<grid, kBS, 0, s>>>(a, w, Sh, Sl, vstride, Y, X, col0);
    }
  };
  switch (T.store) {
    case STORE_F32: run(std::integral_constant<int, STORE_F32>()); break;
    case STORE_F16: run(std::integral_constant<int, STORE_F16>()); break;
    default: run(std::integral_constant<int, STORE_BF16>()); break;
  }
  MG_LAUNCH();
}

// --------------------------------------------------------------------------- coarse stencil
// Hops followed by a site matrix (EPI_CH, EPI_CX_PAY): CTA = site.
struct HopArgs {
  int nc, s0;
  const int* nbr;
  const void* Y;    // links in the level's storage format
  const float* Ys;
  const float2* C;  // X or Xinv
  float2* out;
  const float2* in;
  const float2* x;
  float a;
};

template <int EPI, int ST>
__global__ void __launch_bounds__(256) k_coarse_hop(HopArgs h) {
  extern __shared__ __align__(16) float2 sm[];  // vin[8 nc], t[nc], vx[nc]
  const int nc = h.nc;
  const int s = h.s0 + blockIdx.x;
  float2* vin = sm;
  float2* tv = sm + 8 * nc;
  float2* vx = tv + nc;
  for (int t = threadIdx.x; t < 8 * nc; t += blockDim.x) {
    const int d = t / nc, j = t % nc;
    const float sc = h.Ys[(size_t)s * 8 + d];
    const float2 v = h.in[(size_t)h.nbr[(size_t)s * 8 + d] * nc + j];
    vin[t] = make_float2(sc * v.x, sc * v.y);
  }
  if (EPI == EPI_CX_PAY)
    for (int t = threadIdx.x; t < nc; t += blockDim.x) vx[t] = h.x[(size_t)s * nc + t];
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int rpw = (nc + nw - 1) / nw;
  float2 res[kGemvMaxRows];
  warp_gemv<ST>(static_cast<const char*>(h.Y) + (size_t)s * nc * 8 * nc * link_bytes<ST>(), nc, 8 * nc, vin, w, rpw,
                lane, res);
  if (lane == 0)
#pragma unroll
    for (int r = 0; r < kGemvMaxRows; r++) {
      const int i = w * rpw + r;
      if (r < rpw && i < nc) tv[i] = res[r];
    }
  __syncthreads();
  const float2* src = (EPI == EPI_CX_PAY) ? vx : tv;
  warp_gemv(h.C + (size_t)s * nc * nc, nc, nc, src, w, rpw, lane, res);
  if (lane == 0)
#pragma unroll
    for (int r = 0; r < kGemvMaxRows; r++) {
      const int i = w * rpw + r;
      if (r < rpw && i < nc) {
        if (EPI == EPI_CX_PAY)
          h.out[(size_t)s * nc + i] = make_float2(res[r].x + h.a * tv[i].x, res[r].y + h.a * tv[i].y);
        else
          h.out[(size_t)s * nc + i] = res[r];
      }
    }
}

// Rows of the link blocks without a site matrix: out = L in (+ x): CTA = (site,
// 16 rows), a warp owns two rows.  The links do not depend on the gathered
// vector, so their first steps are in flight before it is: two dependent trips
// to L2 (neighbour index, vector) instead of three.  A single direction reads
// that direction's columns only.
struct RowArgs {
  int nc, s0, lbase;         // link blocks of site s at (s - lbase) nc rows
  int q0, q1;                // pairs of columns of a row to use
  const int* nbr;
  const void* L;
  const float* Ls;           // tile scales, or null
  float2* out;
  const float2* in;
  const float2* x;
  float a;
};
constexpr int kRowSteps = 6;   // link steps in flight per lane and row (192 pairs: Nc = 48)
template <int ST, bool XPAY>
__global__ void __launch_bounds__(256) k_coarse_rows(RowArgs h) {
  extern __shared__ __align__(16) float4 vp[];   // [4 nc] pairs of the gathered vector
  using raw = typename LinkPair<ST>::raw;
  const int nc = h.nc, hc = nc >> 1, K2 = 8 * hc, s = h.s0 + blockIdx.x;
  const int lane = threadIdx.x & 31, i0 = blockIdx.y * 16 + 2 * (threadIdx.x >> 5);
  const char* row[2];
  raw m[kRowSteps][2];
#pragma unroll
  for (int r = 0; r < 2; r++)
    row[r] = static_cast<const char*>(h.L) + ((size_t)(s - h.lbase) * nc + min(i0 + r, nc - 1)) * K2 * sizeof(raw);
  auto load = [&](int qb) {
#pragma unroll
    for (int u = 0; u < kRowSteps; u++)
#pragma unroll
      for (int r = 0; r < 2; r++) {
        const int q = qb + lane + 32 * u;
        m[u][r] = q < h.q1 ? LinkPair<ST>::load(row[r], q) : LinkPair<ST>::zero();
      }
  };
  load(h.q0);
  for (int t = h.q0 + threadIdx.x; t < h.q1; t += blockDim.x) {
    const int d = t / hc, j = t - d * hc;
    const float sc = h.Ls ? h.Ls[(size_t)s * 8 + d] : 1.f;
    const float4 v = reinterpret_cast<const float4*>(h.in + (size_t)h.nbr[(size_t)s * 8 + d] * nc)[j];
    vp[t] = make_float4(sc * v.x, sc * v.y, sc * v.z, sc * v.w);
  }
  __syncthreads();
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  for (int qb = h.q0; qb < h.q1; qb += 32 * kRowSteps) {
    if (qb > h.q0) load(qb);
#pragma unroll
    for (int u = 0; u < kRowSteps; u++) {
      const int q = qb + lane + 32 * u;
      if (q < h.q1) {
        const float4 x = vp[q];
#pragma unroll
        for (int r = 0; r < 2; r++) {
          const float4 l = LinkPair<ST>::decode(m[u][r]);
          acc[2 * r] = fmaf(l.x, x.x, fmaf(-l.y, x.y, fmaf(l.z, x.z, fmaf(-l.w, x.w, acc[2 * r]))));
          acc[2 * r + 1] = fmaf(l.x, x.y, fmaf(l.y, x.x, fmaf(l.z, x.w, fmaf(l.w, x.z, acc[2 * r + 1]))));
        }
      }
    }
  }
  const float t = warp_transpose_sum<4>(acc);   // lane l: value l >> 3 = 2 row + {re, im}
  const float im = __shfl_down_sync(0xffffffffu, t, 8);
  const int r = lane >> 4;
  if ((lane & 15) == 0 && i0 + r < nc) {
    const size_t i = (size_t)s * nc + i0 + r;
    float2 o = make_float2(t, im);
    if (XPAY) {
      const float2 x = h.x[i];
      o = make_float2(x.x + h.a * o.x, x.y + h.a * o.y);
    }
    h.out[i] = o;
  }
}

namespace {
void launch_rows(const RowArgs& h, int sites, int store, bool xpay, cudaStream_t s) {
  const dim3 grid(sites, (h.nc + 15) / 16);
  const size_t sm = sizeof(float2) * 8 * (size_t)h.nc;
  auto run = [&](auto st) {
    constexpr int ST = decltype(st)::value;
    if (xpay)
      k_coarse_rows<ST, true><<<grid, 256, sm, s>>>(h);
    else
      k_coarse_rows<ST, false><<<grid, 256, sm, s>>>(h);
  };
  switch (store) {
    case STORE_F32: run(std::integral_constant<int, kStF32>()); break;
    case STORE_F16: run(std::integral_constant<int, kStF16>()); break;
    default: run(std::integral_constant<int, kStBF16>()); break;
  }
  MG_LAUNCH();
}
}  // namespace

void coarse_folded(const LevelGeom& G, const CoarseOp& C, float* out, const float* in, const float* x, float a,
                   cudaStream_t s) {
  if (!G.eo || !C.A.get()) raise(MG_ERR_STATE, "no folded links on this level");
  RowArgs h;
  h.nc = C.nc;
  h.s0 = h.lbase = G.half;
  h.q0 = 0;
  h.q1 = 4 * C.nc;
  h.nbr = G.d_nbr.as<int>();
  h.L = C.A.get();
  h.Ls = nullptr;
  h.out = (float2*)out;
  h.in = (const float2*)in;
  h.x = (const float2*)x;
  h.a = a;
  launch_rows(h, G.nsites - G.half, STORE_F32, x != nullptr, s);
}

void coarse_hop(const LevelGeom& G, const CoarseOp& C, Epilogue epi, bool use_inv, int s0, int s1, float* out,
                const float* in, const float* x, float a, int dirmask, cudaStream_t s) {
  if (s1 <= s0) return;
  if (epi == EPI_H || epi == EPI_XPAY) {
    const bool single = dirmask != 0xff;
    int d = 0;
    while (single && dirmask >> (d + 1)) d++;
    if (single && dirmask != 1 << d) raise(MG_ERR_ARG, "coarse hops take all directions or one");
    RowArgs r;
    r.nc = C.nc;
    r.s0 = s0;
    r.lbase = 0;
    r.q0 = single ? d * (C.nc / 2) : 0;
    r.q1 = single ? r.q0 + C.nc / 2 : 4 * C.nc;
    r.nbr = G.d_nbr.as<int>();
    r.L = C.Y.get();
    r.Ls = C.Yscale.as<float>();
    r.out = (float2*)out;
    r.in = (const float2*)in;
    r.x = (const float2*)x;
    r.a = a;
    launch_rows(r, s1 - s0, C.store, epi == EPI_XPAY, s);
    return;
  }
  if ((epi != EPI_CH && epi != EPI_CX_PAY) || dirmask != 0xff) raise(MG_ERR_ARG, "no such coarse hop");
  HopArgs h;
  h.nc = C.nc;
  h.s0 = s0;
  h.nbr = G.d_nbr.as<int>();
  h.Y = C.Y.get();
  h.Ys = C.Yscale.as<float>();
  h.C = use_inv ? C.Xinv.as<float2>() : C.X.as<float2>();
  h.out = (float2*)out;
  h.in = (const float2*)in;
  h.x = (const float2*)x;
  h.a = a;
  const size_t sm = sizeof(float2) * 10 * (size_t)C.nc;
  const int nb = s1 - s0;
  auto launch = [&](auto st) {
    constexpr int ST = decltype(st)::value;
    if (epi == EPI_CH)
      k_coarse_hop<EPI_CH, ST><<<nb, 256, sm, s>>>(h);
    else
      k_coarse_hop<EPI_CX_PAY, ST><<<nb, 256, sm, s>>>(h);
  };
  switch (C.store) {
    case STORE_F32: launch(std::integral_constant<int, kStF32>()); break;
    case STORE_F16: launch(std::integral_constant<int, kStF16>()); break;
    default: launch(std::integral_constant<int, kStBF16>()); break;
  }
  MG_LAUNCH();
}

__global__ void __launch_bounds__(256) k_site_mul(int nc, int s0, const float2* __restrict__ C, float2* out,
                                                   const float2* __restrict__ in) {
  extern __shared__ __align__(16) float2 sv[];
  const int s = s0 + blockIdx.x;
  for (int t = threadIdx.x; t < nc; t += blockDim.x) sv[t] = in[(size_t)s * nc + t];
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int rpw = (nc + nw - 1) / nw;
  float2 res[kGemvMaxRows];
  warp_gemv(C + (size_t)s * nc * nc, nc, nc, sv, w, rpw, lane, res);
  if (lane == 0)
#pragma unroll
    for (int r = 0; r < kGemvMaxRows; r++) {
      const int i = w * rpw + r;
      if (r < rpw && i < nc) out[(size_t)s * nc + i] = res[r];
    }
}

void coarse_site_mul(const LevelGeom& G, const CoarseOp& C, bool use_inv, int s0, int s1, float* out, const float* in,
                     cudaStream_t s) {
  (void)G;
  if (s1 <= s0) return;
  const float2* M = use_inv ? C.Xinv.as<float2>() : C.X.as<float2>();
  k_site_mul<<<s1 - s0, 256, sizeof(float2) * C.nc, s>>>(C.nc, s0, M, (float2*)out, (const float2*)in);
  MG_LAUNCH();
}

// --------------------------------------------------------------------------- coarse inverse
// X^{-1} per site in FP64: Gauss-Jordan with row pivoting in place (the columns
// of the inverse replace the eliminated ones; the row exchanges become column
// exchanges at the end), four FMAs per complex element and column.  On the
// augmented matrix [X | 1], with six operations and one thread looking for the
// largest entry, it took three times the FP64 work, the bound here: 512 sites
// of Nc = 48 took 2.23 ms, 0.57 here.
constexpr int kInvThreads = 256;
__global__ void __launch_bounds__(kInvThreads) k_coarse_invert(int nc, const float2* __restrict__ X, float2* Xinv,
                                                               int* flags) {
  extern __shared__ double2 A[];  // [nc][nc]
  __shared__ double2 fac[64];
  __shared__ int perm[64], piv_s;
  __shared__ float wmax[kInvThreads / 32];
  __shared__ double2 pinv_s;
  const int s = blockIdx.x, nn = nc * nc, lane = threadIdx.x & 31;
  const int dq = kInvThreads / nc, dr = kInvThreads % nc, r0 = threadIdx.x / nc, j0 = threadIdx.x % nc;
  float m = 0.f;   // of FP32 entries
  for (int t = threadIdx.x; t < nn; t += kInvThreads) {
    const float2 x = X[(size_t)s * nn + t];
    A[t] = make_double2(x.x, x.y);
    m = fmaxf(m, fabsf(x.x) + fabsf(x.y));
  }
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) wmax[threadIdx.x >> 5] = m;
  __syncthreads();
  for (int col = 0; col < nc; col++) {
    if (threadIdx.x < 32) {
      double best = -1.0;
      int bi = col;
      for (int r = col + lane; r < nc; r += 32) {
        const double2 v = A[r * nc + col];
        const double q = fma(v.x, v.x, v.y * v.y);
        if (q > best) { best = q; bi = r; }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const double ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
      }
      if (lane == 0) {
        float amax = 0.f;
        for (int w = 0; w < kInvThreads / 32; w++) amax = fmaxf(amax, wmax[w]);
        piv_s = perm[col] = bi;
        if (!(sqrt(best) > 1e-12 * (double)amax)) atomicExch(&flags[FLAG_SINGULAR], 1);
        const double2 p = A[bi * nc + col];
        double den = p.x * p.x + p.y * p.y;
        if (den == 0) den = 1;
        pinv_s = make_double2(p.x / den, -p.y / den);
      }
    }
    __syncthreads();
    // rows col and piv exchanged, the pivot row scaled, the column set aside
    const int piv = piv_s;
    const double2 pinv = pinv_s;
    if (threadIdx.x < nc) {
      const int q = threadIdx.x;
      const double2 a = q == col ? make_double2(1.0, 0.0) : A[piv * nc + q];
      if (piv != col) A[piv * nc + q] = A[col * nc + q];
      A[col * nc + q] = make_double2(fma(pinv.x, a.x, -(pinv.y * a.y)), fma(pinv.x, a.y, pinv.y * a.x));
    }
    __syncthreads();
    if (threadIdx.x < nc && threadIdx.x != col) {
      fac[threadIdx.x] = A[threadIdx.x * nc + col];
      A[threadIdx.x * nc + col] = make_double2(0.0, 0.0);
    }
    __syncthreads();
    for (int t = threadIdx.x, r = r0, j = j0; t < nn; t += kInvThreads) {
      if (r != col) {
        const double2 f = fac[r], a = A[col * nc + j];
        double2 v = A[t];
        v.x = fma(-f.x, a.x, fma(f.y, a.y, v.x));
        v.y = fma(-f.x, a.y, fma(-f.y, a.x, v.y));
        A[t] = v;
      }
      r += dq;
      j += dr;
      if (j >= nc) {
        j -= nc;
        r++;
      }
    }
    __syncthreads();
  }
  // column j of the inverse stands where the row exchanges, undone in reverse, put it
  __shared__ int from[64];
  if (threadIdx.x == 0) {
    for (int j = 0; j < nc; j++) from[j] = j;
    for (int col = nc - 1; col >= 0; col--) {
      const int t = from[col];
      from[col] = from[perm[col]];
      from[perm[col]] = t;
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < nn; t += kInvThreads) {
    const double2 v = A[t / nc * nc + from[t % nc]];
    Xinv[(size_t)s * nn + t] = make_float2((float)v.x, (float)v.y);
  }
}

void coarse_invert(const LevelGeom& G, CoarseOp& C, int* flags, cudaStream_t s) {
  const size_t sm = sizeof(double2) * (size_t)C.nc * C.nc;
  MG_CUDA(cudaFuncSetAttribute(k_coarse_invert, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  k_coarse_invert<<<G.nsites, kInvThreads, sm, s>>>(C.nc, C.X.as<float2>(), C.Xinv.as<float2>(), flags);
  MG_LAUNCH();
}

// --------------------------------------------------------------------------- folded links
// One CTA per (odd site o, direction d): A_d(o) = X^{-1}(o) Y_d(o) X^{-1}(o + d).
template <int ST>
__global__ void k_fold_eo(int nc, int half, const int* __restrict__ nbr, const void* __restrict__ Y,
                          const float* __restrict__ Ys, const float2* __restrict__ Xinv, float2* A) {
  extern __shared__ __align__(16) float2 fs[];  // Xo, Yd, Xn, T: 4 nc^2
  const int o = half + blockIdx.x, d = blockIdx.y;
  const int n2 = nc * nc;
  float2* Xo = fs;
  float2* Yd = fs + n2;
  float2* Xn = fs + 2 * n2;
  float2* T = fs + 3 * n2;
  const int nb = nbr[(size_t)o * 8 + d];
  const float sc = Ys[(size_t)o * 8 + d];
  for (int t = threadIdx.x; t < n2; t += blockDim.x) {
    const int i = t / nc, j = t % nc;
    Xo[t] = Xinv[(size_t)o * n2 + t];
    const cx<float> y = sget<ST>(Y, (((size_t)o * nc + i) * 8 + d) * nc + j);
    Yd[t] = make_float2(sc * y.re, sc * y.im);
    Xn[t] = Xinv[(size_t)nb * n2 + t];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < n2; t += blockDim.x) {  // T = Yd Xn
    const int i = t / nc, j = t % nc;
    float re = 0.f, im = 0.f;
    for (int k = 0; k < nc; k++) {
      const float2 a = Yd[i * nc + k], b = Xn[k * nc + j];
      re += a.x * b.x - a.y * b.y;
      im += a.x * b.y + a.y * b.x;
    }
    T[t] = make_float2(re, im);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < n2; t += blockDim.x) {  // A = Xo T
    const int i = t / nc, j = t % nc;
    float re = 0.f, im = 0.f;
    for (int k = 0; k < nc; k++) {
      const float2 a = Xo[i * nc + k], b = T[k * nc + j];
      re += a.x * b.x - a.y * b.y;
      im += a.x * b.y + a.y * b.x;
    }
    A[((((size_t)(o - half)) * nc + i) * 8 + d) * nc + j] = make_float2(re, im);
  }
}

template <int ST>
__global__ void k_cat_links(int nc, int nsites, const void* __restrict__ Y, const float* __restrict__ Ys,
                            const float2* __restrict__ X, float2* A) {
  const size_t total = (size_t)nsites * nc * 9 * nc;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
    const int j = (int)(t % nc);
    const int d = (int)((t / nc) % 9);
    const size_t row = t / ((size_t)9 * nc);  // s * nc + i
    const size_t s = row / nc;
    if (d < 8) {
      const cx<float> y = sget<ST>(Y, (row * 8 + d) * nc + j);
      const float sc = Ys[s * 8 + d];
      A[t] = make_float2(sc * y.re, sc * y.im);
    } else {
      A[t] = X[row * nc + j];
    }
  }
}

void coarse_fold_links(const LevelGeom& G, CoarseOp& C, cudaStream_t s) {
  const int nc = C.nc;
  auto run = [&](auto st) {
    constexpr int ST = decltype(st)::value;
    if (G.eo) {
      const int nodd = G.nsites - G.half;
      C.A.alloc(sizeof(float2) * (size_t)nodd * nc * 8 * nc);
      const size_t sm = sizeof(float2) * 4 * (size_t)nc * nc;
      MG_CUDA(cudaFuncSetAttribute(k_fold_eo<ST>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
      k_fold_eo<ST><<<dim3(nodd, 8), 256, sm, s>>>(nc, G.half, G.d_nbr.as<int>(), C.Y.get(), C.Yscale.as<float>(),
                                                   C.Xinv.as<float2>(), C.A.as<float2>());
    } else {
      C.A.alloc(sizeof(float2) * (size_t)G.nsites * nc * 9 * nc);
      k_cat_links<ST><<<152 * 8, 256, 0, s>>>(nc, G.nsites, C.Y.get(), C.Yscale.as<float>(), C.X.as<float2>(),
                                              C.A.as<float2>());
    }
    MG_LAUNCH();
  };
  switch (C.store) {
    case STORE_F32: run(std::integral_constant<int, STORE_F32>()); break;
    case STORE_F16: run(std::integral_constant<int, STORE_F16>()); break;
    default: run(std::integral_constant<int, STORE_BF16>()); break;
  }
}

// --------------------------------------------------------------------------- 16-bit links
// One CTA per tile (site s = blockIdx.x, block d = blockIdx.y) of an FP32 link
// array [nsites][nc][nb][nc]: scale = largest |Re|, |Im| of the tile (1 for
// an all-zero tile), stored value = link / scale in format ST.
template <int ST>
__global__ void k_quantize_links(int nc, int nb, const float2* __restrict__ in, void* out, float* scale) {
  __shared__ float smax[32];
  __shared__ float sc_s;
  const int s = blockIdx.x, d = blockIdx.y;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int n2 = nc * nc;
  float m = 0.f;
  for (int t = threadIdx.x; t < n2; t += blockDim.x) {
    const int i = t / nc, j = t % nc;
    const float2 z = in[(((size_t)s * nc + i) * nb + d) * nc + j];
    m = fmaxf(m, fmaxf(fabsf(z.x), fabsf(z.y)));
  }
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) smax[wid] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    float v = 0.f;
    for (int q = 0; q < nw; q++) v = fmaxf(v, smax[q]);
    sc_s = v > 0.f ? v : 1.f;
    scale[(size_t)s * nb + d] = sc_s;
  }
  __syncthreads();
  const float inv = 1.f / sc_s;
  for (int t = threadIdx.x; t < n2; t += blockDim.x) {
    const int i = t / nc, j = t % nc;
    const size_t e = (((size_t)s * nc + i) * nb + d) * nc + j;
    const float2 z = in[e];
    sput<ST>(out, e, mkc(z.x * inv, z.y * inv));
  }
}

namespace {
// replaces `buf` ([nsites][nc][nb][nc] FP32) by its 16-bit copy; scales -> `scale`
void quantize_array(DBuf& buf, DBuf& scale, int nsites, int nc, int nb, int store, cudaStream_t s) {
  DBuf q(sizeof(uint32_t) * (size_t)nsites * nc * nb * nc);
  scale.alloc(sizeof(float) * (size_t)nsites * nb);
  const dim3 grid(nsites, nb);
  if (store == STORE_F16)
    k_quantize_links<STORE_F16><<<grid, 256, 0, s>>>(nc, nb, buf.as<float2>(), q.get(), scale.as<float>());
  else
    k_quantize_links<STORE_BF16><<<grid, 256, 0, s>>>(nc, nb, buf.as<float2>(), q.get(), scale.as<float>());
  MG_LAUNCH();
  MG_CUDA(cudaStreamSynchronize(s));
  buf = std::move(q);
}
}  // namespace

void quantize_links(const LevelGeom& G, CoarseOp& C, int store, cudaStream_t s) {
  if (store == STORE_F32) return;
  if (C.store != STORE_F32) raise(MG_ERR_STATE, "coarse links are already quantised");
  if (C.A.get()) raise(MG_ERR_STATE, "quantise the links before folding them");
  quantize_array(C.Y, C.Yscale, G.nsites, C.nc, 8, store, s);
  C.store = store;
}

template <int ST>
__global__ void k_links_abi(int nc, int nsites, const int* __restrict__ lex_of, const void* Y,
                            const float* __restrict__ Ys, const float2* __restrict__ X, double2* Yabi, double2* Xabi) {
  const size_t per = (size_t)9 * nc * nc;
  const size_t total = (size_t)nsites * per;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
    const size_t s = t / per;
    const int r = (int)(t % per);
    const int d = r / (nc * nc), i = (r / nc) % nc, j = r % nc;
    const size_t lex = (size_t)lex_of[s];
    if (d < 8) {
      const cx<float> z = sget<ST>(Y, ((s * nc + i) * 8 + d) * nc + j);
      const double sc = Ys[s * 8 + d];
      Yabi[((lex * 8 + d) * nc + i) * nc + j] = make_double2(sc * z.re, sc * z.im);
    } else {
      const float2 z = X[(s * nc + i) * nc + j];
      Xabi[(lex * nc + i) * nc + j] = make_double2(z.x, z.y);
    }
  }
}

void coarse_links_abi(const LevelGeom& G, const CoarseOp& C, double* Y_abi, double* X_abi, cudaStream_t s) {
  const int nc = C.nc;
  const int* lex = G.d_lex_of.as<int>();
  switch (C.store) {
    case STORE_F32:
      k_links_abi<STORE_F32><<<152 * 8, 256, 0, s>>>(nc, G.nsites, lex, C.Y.get(), C.Yscale.as<float>(),
                                                     C.X.as<float2>(), (double2*)Y_abi, (double2*)X_abi);
      break;
    case STORE_F16:
      k_links_abi<STORE_F16><<<152 * 8, 256, 0, s>>>(nc, G.nsites, lex, C.Y.get(), C.Yscale.as<float>(),
                                                     C.X.as<float2>(), (double2*)Y_abi, (double2*)X_abi);
      break;
    default:
      k_links_abi<STORE_BF16><<<152 * 8, 256, 0, s>>>(nc, G.nsites, lex, C.Y.get(), C.Yscale.as<float>(),
                                                      C.X.as<float2>(), (double2*)Y_abi, (double2*)X_abi);
      break;
  }
  MG_LAUNCH();
}

// --------------------------------------------------------------------------- Philox / packing
__global__ void k_philox_coarse(int nsites, int ndof, const int* lex_of, uint64_t seed, int level, int k, float2* out) {
  const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (t >= (size_t)nsites * ndof) return;
  const int s = (int)(t / ndof), d = (int)(t % ndof);
  const cx<double> z = philox_gauss(seed, level, k, lex_of[s], d);
  out[t] = make_float2((float)z.re, (float)z.im);
}

void philox_coarse_vector(const LevelGeom& G, uint64_t seed, int level, int k, float* out, cudaStream_t s) {
  const size_t n = G.vec_complex();
  k_philox_coarse<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(G.nsites, G.ndof, G.d_lex_of.as<int>(), seed, level, k,
                                                              (float2*)out);
  MG_LAUNCH();
}

__global__ void k_pack_coarse(int nsites, int ndof, const int* lex_of, const double2* abi, float2* v) {
  const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (t >= (size_t)nsites * ndof) return;
  const int s = (int)(t / ndof), d = (int)(t % ndof);
  const double2 z = abi[(size_t)lex_of[s] * ndof + d];
  v[t] = make_float2((float)z.x, (float)z.y);
}

__global__ void k_unpack_coarse(int nsites, int ndof, const int* lex_of, const float2* v, double2* abi) {
  const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (t >= (size_t)nsites * ndof) return;
  const int s = (int)(t / ndof), d = (int)(t % ndof);
  const float2 z = v[t];
  abi[(size_t)lex_of[s] * ndof + d] = make_double2(z.x, z.y);
}

void pack_coarse(const LevelGeom& G, const double* abi, float* v, cudaStream_t s) {
  const size_t n = G.vec_complex();
  k_pack_coarse<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(G.nsites, G.ndof, G.d_lex_of.as<int>(), (const double2*)abi,
                                                            (float2*)v);
  MG_LAUNCH();
}

void unpack_coarse(const LevelGeom& G, const float* v, double* abi, cudaStream_t s) {
  const size_t n = G.vec_complex();
  k_unpack_coarse<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(G.nsites, G.ndof, G.d_lex_of.as<int>(), (const float2*)v,
                                                              (double2*)abi);
  MG_LAUNCH();
}

// --------------------------------------------------------------------------- block Gram-Schmidt
struct GSArgs {
  TArgs a;
  const float* V;       // nv level vectors, vector k at V + k * vstride
  size_t vstride;       // floats between consecutive vectors
  float4* Q;            // [ncoarse][2][nv][L] complex float pairs {re.h, re.l, im.h, im.l}
  int L;                // nb * ndof / 2
};

// The orthonormal vectors do not depend on the vectors' scales, the float-pair
// products do: below about 2^-50 their low halves underflow, above 2^60 the sums
// of squares overflow.  A vector whose largest entry in a block lies outside
// 2^-24 .. 2^24 is multiplied by a power of two there (exactly).
__global__ void k_gs_gather(GSArgs g) {
  __shared__ int s_max[64];   // [chirality][k], bits of the largest |Re|, |Im|
  const int cc = blockIdx.x;
  const int nv = g.a.nv, hd = g.a.ndof / 2, L = g.L;
  const size_t per = (size_t)2 * nv * L;
  if (threadIdx.x < 2 * nv) s_max[threadIdx.x] = 0;
  __syncthreads();
  for (size_t t = threadIdx.x; t < per; t += blockDim.x) {
    const int ck = (int)(t / L), ch = ck / nv;
    const int l = (int)(t % L);
    const int i = l / hd, c = ch * hd + l % hd;
    const int idx = g.a.blockmap[cc * g.a.nb + i];
    const cx<float> z = fget(g.a.fa, g.V + (size_t)(ck % nv) * g.vstride, idx, c);
    g.Q[(size_t)cc * per + t] = make_float4(z.re, 0.f, z.im, 0.f);
    const int m = max(__float_as_int(fabsf(z.re)), __float_as_int(fabsf(z.im)));
    if (m > *(volatile int*)&s_max[ck]) atomicMax(&s_max[ck], m);
  }
  __syncthreads();
  for (int ck = 0; ck < 2 * nv; ck++) {
    const float m = __int_as_float(s_max[ck]);
    if (!(m > 0.f && m <= 3.4e38f) || (m >= 0x1p-24f && m <= 0x1p24f)) continue;
    const int e = ilogbf(m);
    float4* q = g.Q + (size_t)cc * per + (size_t)ck * L;
    for (int l = threadIdx.x; l < L; l += blockDim.x) q[l] = make_float4(ldexpf(q[l].x, -e), 0.f, ldexpf(q[l].z, -e), 0.f);
  }
}

// one CTA per (coarse site, chirality): classical Gram-Schmidt with every
// vector projected twice; breakdown if the norm after projection drops below
// kGSBreakdown of the norm before.  The vectors arrive in FP32, so dependence
// is only resolvable to about 1e-7: the threshold is 1e-6 (the FP64 oracle
// uses 1e-10 on FP64 vectors).
//
// Arithmetic-bound in FP64 (11 ms at the FP64 rate for 512 blocks of 1536 x 24
// x 2 chiralities) and, projected vector by vector, bound by one block barrier
// per inner product (28.8 ms measured).  Here the vector being orthogonalised
// stays in shared memory, all its inner products are taken before one
// reduction, and vectors and sums are float pairs (about 48 bits, twelve FP32
// operations per product against 62 operation slots of an FP64 FMA): 5.6 ms.  Large
// problems run one CTA per SM so that the resident blocks' vectors (590 KB
// each) are re-read from L2.
constexpr double kGSBreakdown = 1e-6;
constexpr int kGSThreads = 512;
constexpr int kGSWarps = kGSThreads / 32;
constexpr size_t kGSFixed = sizeof(df) * (64 * kGSWarps + 64) + 64;   // reduction and coefficients (nv <= 32)

__global__ void __launch_bounds__(kGSThreads) k_block_gs(GSArgs g, int in_smem, int* flags) {
  extern __shared__ __align__(16) unsigned char gsm[];
  df* red = reinterpret_cast<df*>(gsm);            // [2 nv][warp]
  df* coef = red + 64 * kGSWarps;                   // [2 nv]
  float* bc = reinterpret_cast<float*>(coef + 64);  // broadcast values
  float4* wbuf = reinterpret_cast<float4*>(gsm + kGSFixed);
  const int blk = blockIdx.x;  // cc * 2 + ch
  const int nv = g.a.nv, L = g.L;
  float4* Q = g.Q + (size_t)blk * nv * L;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // ||w||^2 (every thread returns with the total in bc[0..1])
  auto norm2 = [&](const float4* w) {
    float h = 0.f, l = 0.f;
    for (int e = threadIdx.x; e < L; e += kGSThreads) {
      const float4 x = w[e];
      df_dot_acc(h, l, df{x.x, x.y}, df{x.x, x.y});
      df_dot_acc(h, l, df{x.z, x.w}, df{x.z, x.w});
    }
    const df t = df_wsum(df_norm(h, l));
    if (lane == 0) red[wid] = t;
    __syncthreads();
    df s = red[0];
#pragma unroll
    for (int q = 1; q < kGSWarps; q++) s = df_add(s, red[q]);
    __syncthreads();
    return s;
  };
  for (int k = 0; k < nv; k++) {
    float4* wk = Q + (size_t)k * L;
    float4* w = in_smem ? wbuf : wk;
    if (in_smem)   // a thread only ever touches its own elements of w
      for (int e = threadIdx.x; e < L; e += kGSThreads) w[e] = wk[e];
    const df n0 = norm2(w);
    for (int pass = 0; pass < 2 && k > 0; pass++) {
      for (int j0 = 0; j0 < k; j0 += 4) {
        float acc[4][4] = {};
        for (int e = threadIdx.x; e < L; e += kGSThreads) {
          float4 q[4];
#pragma unroll
          for (int u = 0; u < 4; u++) q[u] = j0 + u < k ? Q[(size_t)(j0 + u) * L + e] : make_float4(0.f, 0.f, 0.f, 0.f);
          const float4 x = w[e];
          const df xr{x.x, x.y}, xi{x.z, x.w};
#pragma unroll
          for (int u = 0; u < 4; u++) {   // conj(q) x
            const df qr{q[u].x, q[u].y}, qi{q[u].z, q[u].w};
            df_dot_acc(acc[u][0], acc[u][1], qr, xr);
            df_dot_acc(acc[u][0], acc[u][1], qi, xi);
            df_dot_acc(acc[u][2], acc[u][3], qr, xi);
            df_dot_acc(acc[u][2], acc[u][3], df_neg(qi), xr);
          }
        }
        df v[8];
#pragma unroll
        for (int u = 0; u < 4; u++) {
          v[2 * u] = df_norm(acc[u][0], acc[u][1]);
          v[2 * u + 1] = df_norm(acc[u][2], acc[u][3]);
        }
        const df t = warp_transpose_sum<8>(v);   // lane l: value l >> 2
        const int q = 2 * j0 + (lane >> 2);
        if ((lane & 3) == 0 && q < 2 * k) red[q * kGSWarps + wid] = t;
      }
      __syncthreads();
      if (threadIdx.x < 2 * k) {
        df s = red[threadIdx.x * kGSWarps];
#pragma unroll
        for (int q = 1; q < kGSWarps; q++) s = df_add(s, red[threadIdx.x * kGSWarps + q]);
        coef[threadIdx.x] = df_neg(s);
      }
      __syncthreads();
      for (int e = threadIdx.x; e < L; e += kGSThreads) {
        float4 x = w[e];
#pragma unroll 4
        for (int j = 0; j < k; j++) {   // x -= c q
          const float4 q = Q[(size_t)j * L + e];
          const df qr{q.x, q.y}, qi{q.z, q.w}, cr = coef[2 * j], ci = coef[2 * j + 1];
          df_dot_acc(x.x, x.y, cr, qr);
          df_dot_acc(x.x, x.y, df_neg(ci), qi);
          df_dot_acc(x.z, x.w, cr, qi);
          df_dot_acc(x.z, x.w, ci, qr);
        }
        const df re = df_norm(x.x, x.y), im = df_norm(x.z, x.w);
        w[e] = make_float4(re.h, re.l, im.h, im.l);
      }
    }
    const df n1 = norm2(w);
    if (threadIdx.x == 0) {
      const double a = (double)n0.h + (double)n0.l, b = (double)n1.h + (double)n1.l;
      if (!(a > 0) || !(sqrt(b) >= kGSBreakdown * sqrt(a))) atomicExch(&flags[FLAG_GS_BREAKDOWN], 1);
      const double f = b > 0 ? 1.0 / sqrt(b) : 0.0;
      bc[0] = (float)f;
      bc[1] = (float)(f - (double)bc[0]);
    }
    __syncthreads();
    const df f{bc[0], bc[1]};
    for (int e = threadIdx.x; e < L; e += kGSThreads) {
      const float4 x = w[e];
      const df re = df_mul(df{x.x, x.y}, f), im = df_mul(df{x.z, x.w}, f);
      wk[e] = make_float4(re.h, re.l, im.h, im.l);
    }
    __syncthreads();   // q_k of this thread's elements is read by the same thread only; bc is reused
  }
}

// scale per (coarse site, chirality): 1 for FP32 storage, else the largest
// |Re|, |Im| of the tile so that the stored values lie in [-1, 1]
template <int ST>
__global__ void k_gs_scatter(GSArgs g, void* P, float* Ps) {
  __shared__ float smax[2][32];
  __shared__ float scale_s[2];
  const int cc = blockIdx.x;
  const int nv = g.a.nv, hd = g.a.ndof / 2, L = g.L;
  const size_t per = (size_t)2 * nv * L;
  const float4* Qc = g.Q + (size_t)cc * per;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  float m[2] = {0.f, 0.f};
  if (ST != STORE_F32)
    for (size_t t = threadIdx.x; t < per; t += blockDim.x) {
      const int ch = (int)(t / ((size_t)nv * L));
      const float4 z = Qc[t];   // the high halves are the values rounded to FP32
      m[ch] = fmaxf(m[ch], fmaxf(fabsf(z.x), fabsf(z.z)));
    }
  for (int ch = 0; ch < 2; ch++) {
    float v = m[ch];
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (lane == 0) smax[ch][wid] = v;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    float v = 0.f;
    for (int q = 0; q < nw; q++) v = fmaxf(v, smax[threadIdx.x][q]);
    scale_s[threadIdx.x] = (ST == STORE_F32 || v == 0.f) ? 1.f : v;
    Ps[cc * 2 + threadIdx.x] = scale_s[threadIdx.x];
  }
  __syncthreads();
  for (size_t t = threadIdx.x; t < per; t += blockDim.x) {
    const int ch = (int)(t / ((size_t)nv * L));
    const int k = (int)((t / L) % nv);
    const int l = (int)(t % L);
    const int i = l / hd, c = ch * hd + l % hd;
    const float4 z = Qc[t];
    const float inv = 1.f / scale_s[ch];
    sput<ST>(P, ((size_t)(cc * g.a.nb + i) * g.a.ndof + c) * nv + k, mkc(z.x * inv, z.z * inv));
  }
}

void block_orthonormalize(TransferOp& T, const float* const* V, DBuf& scratch, int* flags, cudaStream_t s) {
  GSArgs g;
  g.a = targs(T);
  g.V = V[0];
  g.vstride = (T.nv > 1) ? (size_t)(V[1] - V[0]) : 0;
  for (int k = 2; k < T.nv; k++)
    if ((size_t)(V[k] - V[0]) != k * g.vstride) raise(MG_ERR_ARG, "null vectors must be equally spaced");
  g.L = T.nb * T.fine_ndof / 2;
  const size_t need = sizeof(float4) * (size_t)T.ncoarse * 2 * T.nv * g.L;
  if (scratch.bytes() < need) scratch.alloc(need);
  g.Q = scratch.as<float4>();
  k_gs_gather<<<T.ncoarse, kBS, 0, s>>>(g);
  MG_LAUNCH();
  int dev = 0, optin = 0;
  MG_CUDA(cudaGetDevice(&dev));
  MG_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  size_t sm = kGSFixed + sizeof(float4) * (size_t)g.L;
  const int in_smem = sm <= (size_t)optin;   // a block too large for shared memory works in place
  if (!in_smem) sm = kGSFixed;
  // more than about the L2 capacity of vectors in all: one CTA per SM
  if (need > ((size_t)96 << 20)) sm = std::max<size_t>(sm, (size_t)optin / 2 + 1024);
  MG_CUDA(cudaFuncSetAttribute(k_block_gs, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  k_block_gs<<<T.ncoarse * 2, kGSThreads, sm, s>>>(g, in_smem, flags);
  MG_LAUNCH();
  switch (T.store) {
    case STORE_F32: k_gs_scatter<STORE_F32><<<T.ncoarse, kBS, 0, s>>>(g, T.P.get(), T.Pscale.as<float>()); break;
    case STORE_F16: k_gs_scatter<STORE_F16><<<T.ncoarse, kBS, 0, s>>>(g, T.P.get(), T.Pscale.as<float>()); break;
    default: k_gs_scatter<STORE_BF16><<<T.ncoarse, kBS, 0, s>>>(g, T.P.get(), T.Pscale.as<float>()); break;
  }
  MG_LAUNCH();
}

}  // namespace mg
