// Aggregation-based transfer operators (Sec. 1, Sec. 2.2 of the paper).
//
// P_l is stored as the N orthonormalised test-vector fields of level l.  For
// aggregate A and chirality s (spins 0,1 / 2,3 on the fine level, first and
// second half of the dof on a coarse level), column j of the block
// Q_{A,s} is field j restricted to (A, s); coarse dof (A, s, j) has index s*N + j.
// Aggregates are contiguous index ranges [A*vA, (A+1)*vA) in the site order.
#include "common.cuh"
#include "kernels.h"
#include "tma.cuh"

#include <type_traits>

namespace {

// address of (site x, component f) in a level field: fine [12][V], coarse [V][n]
DD_HD size_t faddr(bool fine, int V, int n, int x, int f) {
  return fine ? (size_t)f * V + x : (size_t)x * n + f;
}


// out(A)[s*N + j] = sum over x in A, f in s of conj(P_j(x, f)) in(x, f).  One CTA per (aggregate, chirality, up to
// three groups of four columns; one column per group in FP64): the N x K by K x C product with K = |A| n/2 in
// chunks of up to 128 rows, copied asynchronously in their storage format into two buffers.  Four warps
// belong to a group; a lane forms a tile of four rows and the group's columns, two rows of K at a time (128 FMAs for
// 8 shared-memory loads at four columns).  The lanes that the ceil(N/4) row tiles leave free and the group's
// warps split K, in a way that depends on the level only, so that a right-hand side has the same bits alone
// and in a batch.  A lane's products of a few chunks run in one chain and are then added to its part, so that neither
// chain is long, and the parts are added with their rounding errors.  An FP16 column on 4^4 aggregates is off by
// 0.87e-7 (8 test vectors) to 1.09e-7 (32) against 64 bits, 20 test vectors 1.07e-7; three chunks in one chain and plain sums of
// the parts gave 1.33e-7 there, one lane per site and a butterfly over the lanes 1.11e-7 (6^4 aggregates 1.79e-7).
// A chunk is whole runs of memory (sites of one component on the fine level, dofs of one site on a coarse one).
// Where those are multiples of 16 bytes (BULK) one lane copies a run of a column with one bulk copy;
// with a copy instruction per pair of elements the copies took two thirds of the issue slots.
// Bound by memory for one right-hand side (P once: 126 MB of FP16 for 20 test vectors on 16^3x32), by FP32 issue
// for many (4 N |A| n FMAs per aggregate and column).
constexpr int RTH = 128;    // threads of a group
constexpr int RKC = 128;    // most K rows of a chunk
constexpr int RNG = 3;      // most groups of a CTA
// columns of a group: one in FP64, where the FMAs bound the kernel and a column tile would only take registers
template <typename T> constexpr int restrict_ct() { return sizeof(T) == 4 ? 4 : 1; }
constexpr int RKP = RKC + 12;  // row pitch of P (elements): a multiple of 16 bytes, the row tiles of a warp on different banks
constexpr int RKB = RKC + 2;   // row pitch of the columns

struct RestrictSmem {
  size_t b, stage, red, bar, total;
};
template <typename T>
DD_HD RestrictSmem restrict_smem(int N, int groups, size_t ps) {
  RestrictSmem L;
  const int TI = (N + 3) / 4;
  L.b = (size_t)N * RKP * ps;
  L.stage = L.b + (size_t)groups * restrict_ct<T>() * RKB * sizeof(cplx<T>);
  L.red = 2 * L.stage;
  L.bar = L.red + (size_t)groups * (RTH / 32) * (32 / TI) * TI * 4 * restrict_ct<T>() * sizeof(cplx<T>);
  L.total = L.bar + 16;
  return L;
}
// rows of a chunk for runs of `run` elements: whole runs, or the largest even part of a longer run (of a multiple of
// 16 bytes for `bulk`); 0: there is none
inline int restrict_chunk(int run, int ps, bool bulk) {
  if (run <= RKC) return (bulk && run * ps % 16) || run % 2 ? 0 : RKC / run * run;
  for (int d = RKC; d >= 2; --d)
    if (run % d == 0 && d % 2 == 0 && !(bulk && d * ps % 16)) return d;
  return 0;
}

// Chunks that run into one chain of a lane's FMAs: a chain of k roundings errs like sqrt(k / 2) of them, so what
// counts is the FMAs of a chain plus the chains of a lane.  One chunk more than makes that least, since every end of a chain
// costs time (16^3x32, 20 test vectors, restriction and interpolation of one column 146 us with one chunk and 142 with
// two, of twelve 524 and 513), as long as it stays below a lane per site (up to 256 lanes), a butterfly over them and the
// warps in a chain.
inline int restrict_flush(int vA, int h, int N, int kch) {
  const int nsub = 32 / ((N + 3) / 4), nch = (vA * h + kch - 1) / kch;
  auto roundings = [&](int f) { return f * kch / (2.0 * nsub) + (double)nch / f; };
  int lanes = 1, levels = 0, f = 1;
  for (; lanes < vA && lanes < 256; lanes *= 2) levels += lanes < 32;
  const double limit = 2.0 * h * ((vA + lanes - 1) / lanes) + 2 * levels + lanes / 32 - 2;
  while (roundings(f + 1) < roundings(f)) ++f;
  return f < nch && roundings(f + 1) <= limit ? f + 1 : f;
}

// (hi, lo) += x without rounding error beyond lo's (Knuth's two-sum)
__device__ __forceinline__ void two_sum_acc(float& hi, float& lo, float x) {
  const float s = __fadd_rn(hi, x), t = __fsub_rn(s, hi);
  lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, t)), __fsub_rn(x, t)));
  hi = s;
}
// the sum that (hi, lo) hold; with an infinite hi, whose rounding error is not a number, hi
__device__ __forceinline__ float two_sum(float hi, float lo) { return isfinite(hi) ? hi + lo : hi; }

// two neighbouring elements of P in shared memory as complex numbers
__device__ __forceinline__ void ld_pair(const __half2* p, cplx<float> a[2]) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  const float2 x = __half22float2(*reinterpret_cast<const __half2*>(&u.x));
  const float2 y = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
  a[0] = cmk<float>(x.x, x.y);
  a[1] = cmk<float>(y.x, y.y);
}
__device__ __forceinline__ void ld_pair(const cplx<float>* p, cplx<float> a[2]) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  a[0] = cmk<float>(v.x, v.y);
  a[1] = cmk<float>(v.z, v.w);
}
__device__ __forceinline__ void ld_pair(const cplx<double>* p, cplx<double> a[2]) {
  a[0] = p[0];
  a[1] = p[1];
}

// kch: K rows of a chunk, run: elements of a run inside a chunk (BULK), flush: chunks that run into one chain of FMAs
template <typename T, typename PS, bool BULK>
__global__ void __launch_bounds__(RNG * RTH, sizeof(T) == 4 ? 2 : 1) k_restrict(
    cplx<T>* __restrict__ out, const cplx<T>* __restrict__ in, const PS* __restrict__ P,
    const float* __restrict__ pscale, Geom gf, bool fine, int n, int N, int nrhs, size_t in_rstride, size_t pstride,
    size_t out_rstride, size_t out_site_stride, int kch, int run, int flush, int* err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int RCT = restrict_ct<T>();
  const int groups = blockDim.x / RTH;
  const int ng = (nrhs + RCT * groups - 1) / (RCT * groups);
  const int r0 = (blockIdx.x % ng) * RCT * groups, C = min(RCT * groups, nrhs - r0);
  const int s = (blockIdx.x / ng) & 1, agg = blockIdx.x / (2 * ng);
  const int V = gf.V, vA = gf.vA, h = n / 2, K = vA * h;
  const RestrictSmem L = restrict_smem<T>(N, groups, sizeof(PS));
  cplx<T>* red = reinterpret_cast<cplx<T>*>(smem_raw + L.red);   // [group][4][RCT][warp][sub][row tile]
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(smem_raw + L.bar);
  const int tid = threadIdx.x, lane = tid & 31, grp = tid / RTH, warp = (tid % RTH) >> 5;
  const int TI = (N + 3) / 4, nsub = 32 / TI, slots = (RTH / 32) * nsub * TI;
  const int sub = lane / TI, ti = lane - sub * TI;       // rows ti, ti + TI, ti + 2 TI, ti + 3 TI
  const int gc = min(RCT, C - grp * RCT);                // columns of the group (none: <= 0)
  const cplx<T>* pin = in + (size_t)r0 * in_rstride;
  // component-major on the fine level (neighbouring rows: neighbouring sites), dof-contiguous on a coarse one
  auto row_addr = [&](int kk) {
    const int q = fine ? fdiv(kk, gf.fvA) : kk / h, r = kk - q * (fine ? vA : h);
    return faddr(fine, V, n, agg * vA + (fine ? r : q), s * h + (fine ? q : r));
  };
  auto copy = [&](int k0, int buf) {
    PS* sA = reinterpret_cast<PS*>(smem_raw + buf * L.stage);                    // [N][RKP]
    cplx<T>* sB = reinterpret_cast<cplx<T>*>(smem_raw + buf * L.stage + L.b);    // [columns][RKB]
    const int kc = min(kch, K - k0);
    if constexpr (BULK) {
      if (tid >= 32) return;
      if (lane == 0) {
        fence_proxy_async_shared();
        mbar_arrive_expect_tx(&bar[buf], (unsigned)(kc * (N * sizeof(PS) + C * sizeof(cplx<T>))));
      }
      __syncwarp();
      for (int q = 0; q < kc; q += run) {
        const size_t a = row_addr(k0 + q);
        for (int j = lane; j < N + C; j += 32) {
          if (j < N) bulk_g2s(sA + j * RKP + q, P + (size_t)j * pstride + a, (unsigned)(run * sizeof(PS)), &bar[buf]);
          else
            bulk_g2s(sB + (j - N) * RKB + q, pin + (size_t)(j - N) * in_rstride + a, (unsigned)(run * sizeof(cplx<T>)),
                     &bar[buf]);
        }
      }
    } else {
      for (int k = tid % RKC; k < kch + (kch & 1); k += RKC) {   // an odd last row's partner is zero
        const bool on = k < kc;
        const size_t a = on ? row_addr(k0 + k) : 0;
        for (int j = tid / RKC; j < N + C; j += groups) {
          if (j < N) cp_async<sizeof(PS)>(sA + j * RKP + k, P + (size_t)j * pstride + a, on);
          else cp_async<sizeof(cplx<T>)>(sB + (j - N) * RKB + k, pin + (size_t)(j - N) * in_rstride + a, on);
        }
      }
      cp_async_commit();
    }
  };
  if (BULK && tid == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
  }
  if (BULK) __syncthreads();
  cplx<T> acc[4][RCT];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int c = 0; c < RCT; ++c) acc[i][c] = czero<T>();
  copy(0, 0);
  int chunk = 0, next = flush - 1;   // the chunk that ends the chain
  bool ok = true, first = true;
  for (int k0 = 0; k0 < K; k0 += kch, ++chunk) {
    const int buf = chunk & 1;
    const bool last = k0 + kch >= K;
    if (!last) copy(k0 + kch, buf ^ 1);
    if constexpr (BULK) {
      ok = mbar_wait_bounded(&bar[buf], (chunk >> 1) & 1);
    } else {
      if (last) cp_async_wait<0>();
      else cp_async_wait<1>();
      __syncthreads();
    }
    const PS* sA = reinterpret_cast<const PS*>(smem_raw + buf * L.stage);
    const cplx<T>* sB = reinterpret_cast<const cplx<T>*>(smem_raw + buf * L.stage + L.b) + grp * RCT * RKB;
    const int kc = (min(kch, K - k0) + 1) / 2;   // pairs
    if (sub < nsub && gc > 0) {
      for (int k = warp * nsub + sub; k < kc; k += (RTH / 32) * nsub) {
        cplx<T> a[4][2];
#pragma unroll
        for (int i = 0; i < 4; ++i) ld_pair(sA + (ti + i * TI < N ? ti + i * TI : 0) * RKP + 2 * k, a[i]);
#pragma unroll
        for (int c = 0; c < RCT; ++c)
          if (c < gc) {   // uniform in the warp
            cplx<T> b[2];
            ld_pair(sB + c * RKB + 2 * k, b);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              cfmac(acc[i][c], a[i][0], b[0]);
              cfmac(acc[i][c], a[i][1], b[1]);
            }
          }
      }
      if (chunk == next || last) {
        cplx<T>* mine = red + (size_t)grp * 4 * RCT * slots + (warp * nsub + sub) * TI + ti;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int c = 0; c < RCT; ++c)
            if (c < gc) {
              cplx<T>& m = mine[(i * RCT + c) * slots];
              m = first ? acc[i][c] : m + acc[i][c];
              acc[i][c] = czero<T>();
            }
        first = false;
        next += flush;
      }
    }
    if (!BULK) {
      __syncthreads();
    } else if (!__syncthreads_and(ok ? 1 : 0)) {   // a copy did not land in time: flag it, wait for those in flight
      if (tid == 0) {                              // (bounded) and leave
        atomicExch(err, 2);
        mbar_wait_bounded(&bar[buf], (chunk >> 1) & 1);
        if (!last) mbar_wait_bounded(&bar[buf ^ 1], ((chunk + 1) >> 1) & 1);
      }
      return;
    }
  }
  cplx<T>* po = out + (size_t)r0 * out_rstride + (size_t)gf.csite[agg] * out_site_stride + (size_t)s * N;
  const T sc = pscale ? T(pscale[agg * 2 + s]) : T(1);
  // The parts in four chains, FP32 with the rounding errors, then the chains in order: by one thread, or, where there
  // are threads enough, by a lane per chain in the same order (the same bits).
  auto add = [&](cplx<T>& hi, cplx<T>& lo, const cplx<T>& h) {
    if constexpr (sizeof(T) == 4) {
      two_sum_acc(hi.re, lo.re, h.re);
      two_sum_acc(hi.im, lo.im, h.im);
    } else {
      hi = hi + h;
    }
  };
  auto part = [&](int e) {
    const int c = e / N, i = e - c * N;
    return red + ((size_t)(c / RCT) * 4 * RCT + i / TI * RCT + c % RCT) * slots + i % TI;
  };
  auto store = [&](int e, cplx<T> hi, const cplx<T>& lo) {
    if constexpr (sizeof(T) == 4) hi = cmk(two_sum(hi.re, lo.re), two_sum(hi.im, lo.im));
    po[(size_t)(e / N) * out_rstride + e % N] = sc * hi;
  };
  const int parts = (RTH / 32) * nsub;
  if (4 * N * C <= (int)blockDim.x) {
    if (tid >= ((4 * N * C + 31) & ~31)) return;   // whole warps
    const int e = tid >> 2;
    cplx<T> hi = czero<T>(), lo = czero<T>();
    if (e < N * C)
      for (int q = tid & 3; q < parts; q += 4) add(hi, lo, part(e)[q * TI]);
    const cplx<T> h1 = hi, l1 = lo;
#pragma unroll
    for (int u = 1; u < 4; ++u) {
      const int from = (lane & ~3) | u;
      const cplx<T> h = cmk(__shfl_sync(0xffffffffu, h1.re, from), __shfl_sync(0xffffffffu, h1.im, from));
      add(hi, lo, h);
      if constexpr (sizeof(T) == 4)
        lo = lo + cmk(__shfl_sync(0xffffffffu, l1.re, from), __shfl_sync(0xffffffffu, l1.im, from));
    }
    if (e < N * C && (tid & 3) == 0) store(e, hi, lo);
    return;
  }
  for (int e = tid; e < N * C; e += blockDim.x) {
    const cplx<T>* r = part(e);
    cplx<T> hi[4] = {czero<T>(), czero<T>(), czero<T>(), czero<T>()}, lo[4] = {czero<T>(), czero<T>(), czero<T>(), czero<T>()};
    for (int q = 0; q < parts; q += 4)
#pragma unroll
      for (int u = 0; u < 4; ++u) add(hi[u], lo[u], r[(q + u) * TI]);
#pragma unroll
    for (int u = 1; u < 4; ++u) {
      add(hi[0], lo[0], hi[u]);
      lo[0] = lo[0] + lo[u];
    }
    store(e, hi[0], lo[0]);
  }
}

template <typename T, typename PS>
__global__ void k_prolong(cplx<T>* __restrict__ out, const cplx<T>* __restrict__ in, const PS* __restrict__ P,
                          const float* __restrict__ pscale, Geom gf, bool fine, int n, int N,
                          size_t out_rstride, size_t in_rstride, size_t pstride, bool accumulate) {
  // blockIdx.x: elements of a component (fine) or of all sites (coarse); blockIdx.z: component (fine)
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int V = gf.V;
  if (t >= (fine ? V : V * n)) return;
  const int x = fine ? t : t / n, f = fine ? (int)blockIdx.z : t - x * n;
  const int cs = gf.csite[fdiv(x, gf.fvA)];
  const int s = f < n / 2 ? 0 : 1;
  const cplx<T>* pc = in + (size_t)blockIdx.y * in_rstride + (size_t)cs * (2 * N) + s * N;
  cplx<T> acc = czero<T>();
  const size_t a = faddr(fine, V, n, x, f);
  for (int j = 0; j < N; ++j) cfma(acc, ld_cplx(P, (size_t)j * pstride + a), pc[j]);
  if (pscale) acc = T(pscale[(x / gf.vA) * 2 + s]) * acc;
  cplx<T>* po = out + (size_t)blockIdx.y * out_rstride + a;
  *po = accumulate ? *po + acc : acc;
}

// Galerkin products: columns of P^+ (term of D P), for C <= 8 columns of one launch.
//   out[c][site of A][s*N + i] = sum over x in A, f in s of conj(P_i(x, f)) tmp_c(x, f)
// A term of a hop that leaves the aggregate is nonzero on one face of it only, and only those sites are read
// (tmp is not even written elsewhere): of 4^4 aggregates a quarter, for eight of the nine terms.  FP32 products are summed
// in FP32 over two chunks and from there on with their rounding errors (pairs), and rounded to FP32 once: against
// FP64 the blocks of 16^3x32 are off by 3.9e-8 (5.1e-8 with plain sums).
// One CTA per (aggregate, chirality): the N x K by K x C product with K staged in chunks, each lane a 4 x 4
// tile of the result (64 FMAs for 8 shared-memory loads), the lanes that N x C does not need and the warps
// splitting K (summed at the end in a fixed order).
// Replaces k_restrict with one right-hand side per CTA, which read all of P again for each: the nine terms and
// 40 columns of 16^3x32 with 20 test vectors took 24.3 ms there and take 4.9 ms here, and the second level's
// (4^3x8 sites, 28 test vectors) 4.2 and 0.85 ms.
constexpr int GT = 256;    // threads
constexpr int GKC = 64;    // K rows per staged chunk
constexpr int GCMAX = 8;   // columns per launch

constexpr int GFLUSH = 2;  // chunks whose products run into one accumulator

struct GalerkinSmem {
  size_t red, list, total;
};
// shares of a chunk's rows within a warp: as many as its lanes hold tiles, and no more than there are rows
DD_HD int galerkin_nsub(int tiles) {
  return 32 / tiles < GKC / (GT / 32) ? 32 / tiles : GKC / (GT / 32);
}
DD_HD GalerkinSmem galerkin_smem(int N, int C, int vA, size_t cs) {
  GalerkinSmem L;
  const int tiles = ((N + 3) / 4) * ((C + 3) / 4);
  const int nsub = galerkin_nsub(tiles);
  L.red = (((size_t)GKC * ((N | 1) + (C | 1)) * cs) + 15) & ~size_t(15);
  L.list = L.red + (size_t)(cs == sizeof(cplx<float>) ? 2 : 1) * (GT / 32) * nsub * tiles * 16 * cs;
  L.total = L.list + (size_t)vA * sizeof(int);
  return L;
}

template <typename T>
__global__ void __launch_bounds__(GT) k_galerkin(cplx<double>* __restrict__ out, const cplx<T>* __restrict__ tmp,
                                                 const cplx<T>* __restrict__ P, Geom gf, bool fine, int n, int N, int C,
                                                  size_t tmp_rstride, size_t pstride, size_t out_rstride,
                                                 size_t out_site_stride, int sel, int sel_mu) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int wcount[GT / 32];
  __shared__ int nsites;
  const int agg = blockIdx.x, s = blockIdx.y;
  const int V = gf.V, vA = gf.vA, h = n / 2;
  const int NP = N | 1, CP = C | 1;
  cplx<T>* sA = reinterpret_cast<cplx<T>*>(smem_raw);   // [GKC][NP]
  cplx<T>* sB = sA + (size_t)GKC * NP;                  // [GKC][CP]
  const GalerkinSmem L = galerkin_smem(N, C, vA, sizeof(cplx<T>));
  cplx<T>* red = reinterpret_cast<cplx<T>*>(smem_raw + L.red);   // [16][warp][sub][tile] partial tiles
  int* list = reinterpret_cast<int*>(smem_raw + L.list);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // the sites of the aggregate that the term reaches, in site order
  if (tid == 0) nsites = 0;
  for (int x0 = 0; x0 < vA; x0 += GT) {
    bool take = x0 + tid < vA;
    if (take && sel != SEL_AGG_SELF) {
      int c[4];
      geom_coords(gf, agg * vA + x0 + tid, c);
      take = !hop_internal(gf, c, sel_mu, sel == SEL_AGG_FWD ? +1 : -1, gf.fA);
    }
    const unsigned m = __ballot_sync(0xffffffffu, take);
    if (lane == 0) wcount[warp] = __popc(m);
    __syncthreads();
    int at = nsites;
    for (int w = 0; w < warp; ++w) at += wcount[w];
    if (take) list[at + __popc(m & ((1u << lane) - 1))] = x0 + tid;
    __syncthreads();
    if (tid == 0)
      for (int w = 0; w < GT / 32; ++w) nsites += wcount[w];
    __syncthreads();
  }
  const int nS = nsites, K = nS * h;
  const int TI = (N + 3) / 4, TC = (C + 3) / 4, tiles = TI * TC, nsub = galerkin_nsub(tiles);
  const int sub = lane / tiles, tile = lane - sub * tiles;
  const int i0 = 4 * (tile % TI), c0 = 4 * (tile / TI);
  cplx<T> acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[i][c] = czero<T>();
  // row tid % GKC of a chunk, columns tid / GKC + 4 q of [P | tmp], the next chunk on its way during the product
  constexpr int NL = (32 + GCMAX + GT / GKC - 1) / (GT / GKC);
  const int kr = tid % GKC, j0 = tid / GKC;
  cplx<T> v[NL];
  auto fetch = [&](int k0) {
    const int kk = k0 + kr;
    if (kk < K) {
      // component-major on the fine level (neighbouring rows: neighbouring sites), dof-contiguous on a coarse one
      const int q = fine ? kk / nS : kk / h, r = kk - q * (fine ? nS : h);
      const size_t a = faddr(fine, V, n, agg * vA + list[fine ? r : q], s * h + (fine ? q : r));
#pragma unroll
      for (int e = 0; e < NL; ++e) {
        const int j = j0 + e * (GT / GKC);
        if (j < N) v[e] = P[(size_t)j * pstride + a];
        else if (j < N + C) v[e] = tmp[(size_t)(j - N) * tmp_rstride + a];
      }
    } else {
#pragma unroll
      for (int e = 0; e < NL; ++e) v[e] = czero<T>();
    }
  };
  cplx<T>* mine = red + (warp * nsub + sub) * tiles + tile;
  const int slots = (GT / 32) * nsub * tiles;
  fetch(0);
  int chunk = 0;
  for (int k0 = 0; k0 < K; k0 += GKC, ++chunk) {
#pragma unroll
    for (int e = 0; e < NL; ++e) {
      const int j = j0 + e * (GT / GKC);
      if (j < N) sA[kr * NP + j] = v[e];
      else if (j < N + C) sB[kr * CP + j - N] = v[e];
    }
    __syncthreads();
    if (k0 + GKC < K) fetch(k0 + GKC);
    const int kc = min(GKC, K - k0);
    if (sub < nsub) {
      for (int k = warp * nsub + sub; k < kc; k += (GT / 32) * nsub) {
        cplx<T> a[4], b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = i0 + i < N ? sA[k * NP + i0 + i] : czero<T>();
#pragma unroll
        for (int c = 0; c < 4; ++c) b[c] = c0 + c < C ? sB[k * CP + c0 + c] : czero<T>();
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            cfmac(acc[i][c], a[i], b[c]);
          }
      }
      // long FP32 sums in parts: their rounding errors do not add up along the whole of K
      if ((sizeof(T) == 4 && chunk % GFLUSH == GFLUSH - 1) || k0 + GKC >= K) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            cplx<T>& m = mine[(4 * i + c) * slots];
            if constexpr (sizeof(T) == 4) {
              cplx<T>& e = mine[(16 + 4 * i + c) * slots];
              cplx<T> hi = chunk < GFLUSH ? acc[i][c] : m, lo = chunk < GFLUSH ? czero<T>() : e;
              if (chunk >= GFLUSH) {
                two_sum_acc(hi.re, lo.re, acc[i][c].re);
                two_sum_acc(hi.im, lo.im, acc[i][c].im);
              }
              m = hi;
              e = lo;
            } else {
              m = acc[i][c];
            }
            acc[i][c] = czero<T>();
          }
      }
    }
    __syncthreads();
  }
  cplx<double>* po = out + (size_t)gf.csite[agg] * out_site_stride + (size_t)s * N;
  for (int e = tid; e < N * C; e += GT) {
    const int c = e / N, i = e - c * N;
    const cplx<T>* r = red + (4 * (i % 4) + c % 4) * slots + (c / 4) * TI + i / 4;
    if constexpr (sizeof(T) == 4) {
      cplx<T> hi = czero<T>(), lo = czero<T>();
      for (int q = 0; K > 0 && q < (GT / 32) * nsub; ++q) {
        const cplx<T> h = r[q * tiles], l = r[16 * slots + q * tiles];
        two_sum_acc(hi.re, lo.re, h.re);
        two_sum_acc(hi.im, lo.im, h.im);
        lo = lo + l;
      }
      po[(size_t)c * out_rstride + i] = cmk((double)two_sum(hi.re, lo.re), (double)two_sum(hi.im, lo.im));
      continue;
    }
    cplx<T> t[4] = {czero<T>(), czero<T>(), czero<T>(), czero<T>()};   // the parts in four chains
    for (int q = 0; K > 0 && q < (GT / 32) * nsub; q += 4)
#pragma unroll
      for (int u = 0; u < 4; ++u) t[u] = t[u] + r[(q + u) * tiles];
    po[(size_t)c * out_rstride + i] = ccast<double>((t[0] + t[1]) + (t[2] + t[3]));
  }
}

// CGS2 of the N test vectors restricted to (aggregate, chirality), in column order.  One CTA per
// (aggregate, chirality); the column in work stays in shared memory (SW) while it is orthogonalised, the earlier
// ones are read from L2 or HBM, and both run through the elements as memory holds them.
// Bound by the FP64 rate: 16 FMAs per element and pair of columns, 4.8 G of them for 20 columns on 16^3x32,
// 9.1 ms, measured 11.4 (21.8 before).  Eight dot products are reduced together by lanes that share the values out as they fold (16 additions
// per lane instead of 80, and the warps' sums are added by one warp instead of all).
constexpr int OT = 128;   // threads

// sum 16 values per thread over the warp: lane l returns value l / 2
__device__ __forceinline__ double warp_fold16(double* v, int lane) {
#pragma unroll
  for (int w = 8, off = 16; w >= 1; w >>= 1, off >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int k = 0; k < w; ++k) {
      const double keep = up ? v[k + w] : v[k], send = up ? v[k] : v[k + w];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

template <bool SW>
__global__ void __launch_bounds__(OT) k_orthonormalise(cplx<double>* __restrict__ P, Geom g, bool fine, int n, int N,
                                                       size_t pstride, int* err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double sh[OT / 32][16];
  __shared__ cplx<double> hs[64];
  __shared__ double tot;
  cplx<double>* sw = reinterpret_cast<cplx<double>*>(smem_raw);   // [ne] the column in work
  const int agg = blockIdx.x;
  const int s = blockIdx.y;
  const int h = n / 2;
  const int ne = g.vA * h;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // element e of the block: fine fields by component, then site; coarse fields by site, then dof
  auto addr = [&](int e) -> size_t {
    if (fine) {
      const int f = fdiv(e, g.fvA);
      return (size_t)(s * h + f) * g.V + (size_t)agg * g.vA + (e - f * g.vA);
    }
    const int x = e / h;
    return (size_t)(agg * g.vA + x) * n + s * h + (e - x * h);
  };
  auto cta_norm2 = [&](const cplx<double>* w) {
    double a = 0.0;
    for (int e = threadIdx.x; e < ne; e += OT) cnorm2_acc(a, SW ? sw[e] : w[addr(e)]);
    for (int off = 16; off >= 1; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
    __syncthreads();
    if (lane == 0) sh[warp][0] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w2 = 0; w2 < OT / 32; ++w2) t += sh[w2][0];
      tot = t;
    }
    __syncthreads();
    return tot;
  };
  for (int j = 0; j < N; ++j) {
    cplx<double>* w = P + (size_t)j * pstride;
    if (SW)
      for (int e = threadIdx.x; e < ne; e += OT) sw[e] = w[addr(e)];   // read back by the same thread
    const double n0 = cta_norm2(w);
    for (int pass = 0; pass < 2 && j > 0; ++pass) {
      for (int i0 = 0; i0 < j; i0 += 8) {
        double acc[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) acc[k] = 0.0;
        for (int e = threadIdx.x; e < ne; e += OT) {
          const size_t a = addr(e);
          const cplx<double> we = SW ? sw[e] : w[a];
#pragma unroll
          for (int ii = 0; ii < 8; ++ii)
            if (i0 + ii < j) cdotc_acc(acc[2 * ii], acc[2 * ii + 1], P[(size_t)(i0 + ii) * pstride + a], we);
        }
        const double v = warp_fold16(acc, lane);
        if ((lane & 1) == 0) sh[warp][lane >> 1] = v;
        __syncthreads();
        if (threadIdx.x < 16 && i0 + (threadIdx.x >> 1) < j) {
          double t = 0.0;
          for (int w2 = 0; w2 < OT / 32; ++w2) t += sh[w2][threadIdx.x];
          reinterpret_cast<double*>(hs)[2 * i0 + threadIdx.x] = t;
        }
        __syncthreads();
      }
      for (int e = threadIdx.x; e < ne; e += OT) {
        const size_t a = addr(e);
        cplx<double> we = SW ? sw[e] : w[a];
#pragma unroll 4
        for (int i = 0; i < j; ++i) cfma(we, cmk(-hs[i].re, -hs[i].im), P[(size_t)i * pstride + a]);
        if (SW) sw[e] = we;
        else w[a] = we;
      }
      __syncthreads();   // hs is read before the second pass writes it
    }
    const double nrm = sqrt(cta_norm2(w));
    if (!(nrm > 1e-12 * sqrt(n0)) || n0 == 0.0) {
      if (threadIdx.x == 0) atomicExch(err, 1);
      return;
    }
    const double inv = 1.0 / nrm;
    for (int e = threadIdx.x; e < ne; e += OT) {
      const size_t a = addr(e);
      w[a] = inv * (SW ? sw[e] : w[a]);
    }
    // every element of a column is written and read by one thread of the CTA: no barrier
  }
}

// FP16 copy of P with one scale per (aggregate, chirality): s = float(max |re|, |im|)
// over the N columns restricted to (A, s), q = RNE_half(x / s), x / s as the product with the reciprocal
// (1.5 units in the last FP64 place before the rounding to FP16) and the maximum on the bits: an FP64 division
// and comparison per value bound this kernel by the FP64 rate (1.2 ms for 20 columns on 16^3x32, now 0.33).
__global__ void k_p_to_half(__half2* __restrict__ Ph, float* __restrict__ pscale, const cplx<double>* __restrict__ P,
                            Geom g, bool fine, int n, int N, size_t pstride) {
  __shared__ unsigned long long sh[32];
  __shared__ double rs;
  const int agg = blockIdx.x, s = blockIdx.y, h = n / 2;
  const int ne = g.vA * h;
  const int V = g.V;
  // element e as memory holds it: by component, then site (fine), by site, then dof (coarse)
  auto addr = [&](int j, int e) -> size_t {
    const int q = fine ? fdiv(e, g.fvA) : e / h, r = e - q * (fine ? g.vA : h);
    return (size_t)j * pstride + faddr(fine, V, n, agg * g.vA + (fine ? r : q), s * h + (fine ? q : r));
  };
  unsigned long long mx = 0ull;
  for (int j = 0; j < N; ++j)
    for (int e = threadIdx.x; e < ne; e += blockDim.x) {
      const cplx<double> v = P[addr(j, e)];
      mx = max(mx, max(abs_bits(v.re), abs_bits(v.im)));
    }
  for (int off = 16; off >= 1; off >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, off));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) mx = max(mx, sh[w]);
    const double m = __longlong_as_double((long long)mx);
    const float sf = m > 0.0 ? (float)m : 1.0f;
    pscale[agg * 2 + s] = sf;
    rs = 1.0 / (double)sf;
  }
  __syncthreads();
  const double r = rs;
  for (int j = 0; j < N; ++j)
    for (int e = threadIdx.x; e < ne; e += blockDim.x) {
      const size_t a = addr(j, e);
      const cplx<double> v = P[a];
      Ph[a] = __halves2half2(__double2half(v.re * r), __double2half(v.im * r));
    }
}

}  // namespace

namespace dd {

void p_to_half(__half2* Ph, float* pscale, const cplx<double>* P, const Geom& g, bool fine, int n, int N,
               cudaStream_t st) {
  count_launch();
  k_p_to_half<<<dim3(g.nAgg, 2), 256, 0, st>>>(Ph, pscale, P, g, fine, n, N, (size_t)g.V * n);
}

template <typename T>
cudaError_t restrict_op(cplx<T>* out, const cplx<T>* in, const cplx<T>* P, const Geom& gf, const Geom& gc, bool fine,
                        int n, int N, int nrhs, size_t in_rstride, size_t out_rstride, size_t out_site_stride, int* err,
                        cudaStream_t st, const __half2* Ph, const float* pscale, int tc_ks) {
  if constexpr (sizeof(T) == 4) {
    // FP16 P: the tensor-core kernel (P read once per batch) where the autotuner chose it
    if (Ph && tc_ks > 0) {
      if (restrict_tc(out, in, Ph, pscale, gf, fine, n, N, nrhs, in_rstride, out_rstride, out_site_stride, tc_ks,
                      st) == cudaSuccess)
        return cudaSuccess;
      cudaGetLastError();
    }
  }
  const size_t pstride = (size_t)gf.V * n;
  auto launch = [&](auto* Ps, const float* scale) {
    using PS = std::remove_const_t<std::remove_pointer_t<decltype(Ps)>>;
    constexpr int RCT = restrict_ct<T>();
    // bulk copies: whole runs of multiples of 16 bytes at 16-byte aligned addresses, in P and in the columns (the
    // smaller elements decide)
    const int run = fine ? gf.vA : n / 2;
    const size_t pb = sizeof(PS);
    const bool aligned = (uintptr_t)in % 16 == 0 && (uintptr_t)Ps % 16 == 0 && in_rstride * sizeof(cplx<T>) % 16 == 0 &&
                         pstride * pb % 16 == 0 && (fine ? (size_t)gf.V : (size_t)n) * pb % 16 == 0;
    int kch = aligned && err ? restrict_chunk(run, (int)pb, true) : 0;
    const bool bulk = kch > 0 && run * pb % 16 == 0;
    if (!bulk) kch = RKC;
    // groups of columns that share a copy of P, as far as shared memory takes them
    int groups = (nrhs + RCT - 1) / RCT;
    if (groups > RNG) groups = RNG;
    while (groups > 1 && restrict_smem<T>(N, groups, pb).total > 110 * 1024) --groups;
    const unsigned grid = (unsigned)gf.nAgg * 2u * (unsigned)((nrhs + RCT * groups - 1) / (RCT * groups));
    auto kernel = bulk ? k_restrict<T, PS, true> : k_restrict<T, PS, false>;
    static DeviceOnce once[2];
    raise_smem_limit(once[bulk], (const void*)kernel);
    count_launch();
    kernel<<<grid, groups * RTH, restrict_smem<T>(N, groups, pb).total, st>>>(
        out, in, Ps, scale, gf, fine, n, N, nrhs, in_rstride, pstride, out_rstride, out_site_stride, kch,
        run < kch ? run : kch, restrict_flush(gf.vA, n / 2, N, kch), err);
    return cudaPeekAtLastError();
  };
  if constexpr (sizeof(T) == 4) {
    if (Ph) return launch(Ph, pscale);
  }
  return launch(P, (const float*)nullptr);
}

template <typename T>
void prolong_op(cplx<T>* out, const cplx<T>* in, const cplx<T>* P, const Geom& gf, const Geom& gc, bool fine, int n,
                int N, int nrhs, size_t out_rstride, size_t in_rstride, bool accumulate, cudaStream_t st,
                const __half2* Ph, const float* pscale, int batch) {
  if constexpr (sizeof(T) == 4) {
    // FP16 P: one CTA per aggregate for the whole batch (P read once) where the autotuner chose it
    if (Ph && batch) {
      if (prolong_batch(out, in, Ph, pscale, gf, fine, n, N, nrhs, out_rstride, in_rstride, accumulate, st) ==
          cudaSuccess)
        return;
      cudaGetLastError();
    }
  }
  const size_t pstride = (size_t)gf.V * n;
  const dim3 grid(div_up(fine ? (size_t)gf.V : (size_t)gf.V * n, 128), nrhs, fine ? n : 1);
  count_launch();
  if constexpr (sizeof(T) == 4) {
    if (Ph) {
      k_prolong<float, __half2><<<grid, 128, 0, st>>>(
          out, in, Ph, pscale, gf, fine, n, N, out_rstride, in_rstride, pstride, accumulate);
      return;
    }
  }
  k_prolong<T, cplx<T>><<<grid, 128, 0, st>>>(out, in, P, nullptr, gf, fine, n, N,
                                                                       out_rstride, in_rstride, pstride, accumulate);
}

cudaError_t orthonormalise(cplx<double>* P, const Geom& g, bool fine, int n, int N, int* err, cudaStream_t st) {
  const size_t pstride = (size_t)g.V * n;
  const size_t sm = (size_t)g.vA * (n / 2) * sizeof(cplx<double>);   // the column in work
  static DeviceOnce once;
  raise_smem_limit(once, (const void*)k_orthonormalise<true>);
  count_launch();
  if (sm <= 200 * 1024)
    k_orthonormalise<true><<<dim3(g.nAgg, 2), OT, sm, st>>>(P, g, fine, n, N, pstride, err);
  else
    k_orthonormalise<false><<<dim3(g.nAgg, 2), OT, 0, st>>>(P, g, fine, n, N, pstride, err);
  return cudaPeekAtLastError();
}

int galerkin_cols() { return GCMAX; }

// FP64 with one or two test vectors: a 4 x 4 tile is mostly padding and a chunk of 64 rows too little in flight; the
// rebuild of 24^3x48 with two takes 40.8 ms with these products and 24.6 with k_restrict, with four 53.9 and 68.5
// (16^3x32: 8.4 and 5.6 ms with two, 11.0 and 14.2 with four, 73.6 and 128 with twenty).
template <typename T>
bool galerkin_fits(int N, int C, int vA) {
  if (sizeof(T) == 8 && N <= 2) return false;
  return C >= 1 && C <= GCMAX && N <= 32 && galerkin_smem(N, C, vA, sizeof(cplx<T>)).total <= 200 * 1024;
}

template <typename T>
cudaError_t galerkin_restrict(cplx<double>* out, const cplx<T>* tmp, const cplx<T>* P, const Geom& gf, const Geom& gc,
                              bool fine, int n, int N, int C, size_t tmp_rstride, size_t out_rstride,
                              size_t out_site_stride, int sel, int sel_mu, cudaStream_t st) {
  const size_t sm = galerkin_smem(N, C, gf.vA, sizeof(cplx<T>)).total;
  if (!galerkin_fits<T>(N, C, gf.vA)) return cudaErrorInvalidValue;
  static DeviceOnce once;
  raise_smem_limit(once, (const void*)k_galerkin<T>);
  count_launch();
  k_galerkin<T><<<dim3(gf.nAgg, 2), GT, sm, st>>>(out, tmp, P, gf, fine, n, N, C, tmp_rstride, (size_t)gf.V * n,
                                                  out_rstride, out_site_stride, sel, sel_mu);
  return cudaPeekAtLastError();
}

#define INST(T)                                                                                                  \
  template cudaError_t restrict_op<T>(cplx<T>*, const cplx<T>*, const cplx<T>*, const Geom&, const Geom&, bool, int, \
                                      int, int, size_t, size_t, size_t, int*, cudaStream_t, const __half2*,       \
                                      const float*, int);                                                        \
  template void prolong_op<T>(cplx<T>*, const cplx<T>*, const cplx<T>*, const Geom&, const Geom&, bool, int, int,  \
                              int, size_t, size_t, bool, cudaStream_t, const __half2*, const float*, int);   \
  template bool galerkin_fits<T>(int, int, int);                                                                 \
  template cudaError_t galerkin_restrict<T>(cplx<double>*, const cplx<T>*, const cplx<T>*, const Geom&, const Geom&, bool, \
                                            int, int, int, size_t, size_t, size_t, int, int, cudaStream_t);
INST(float)
INST(double)
#undef INST

}  // namespace dd
