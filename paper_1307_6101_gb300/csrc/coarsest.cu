// Coarsest-level solve (Sec. 3 of the paper: odd-even preconditioned GMRES to
// relative accuracy epsilon) as one persistent kernel per right-hand side on a
// thread-block cluster.
//
// With D = [[S_ee, D_eo], [D_oe, S_oo]] and S_oo inverted at setup, GMRES(m)
// runs on Dhat = S_ee - D_eo S_oo^{-1} D_oe for bhat_e = b_e - D_eo S_oo^{-1} b_o;
// afterwards z_o = S_oo^{-1} (b_o - D_oe z_e).  CTA q of the cluster owns a
// contiguous slice of the even sites and of the odd sites.  It keeps its rows
// of the Krylov basis in shared memory; neighbour values are read from the
// owning CTA's shared memory (distributed shared memory), dot products are
// summed from per-CTA partials in rank order (identical in every CTA), and the
// Givens updates are computed redundantly by every CTA, so no CTA waits on a
// broadcast.  Cluster barriers separate the phases.  All loops are bounded by
// max_cycles * m.  Stopping rules are those of the host-driven solver: |g_{j+1}|
// <= tol ||bhat|| inside a cycle, the recomputed residual between cycles.
//
// Resident variant (NR > 0: FP32 arithmetic on FP16 blocks, one even and one odd
// site per CTA): the operator does not change during the solve, so each CTA
// loads it once -- the rows of its odd site's 8 hop blocks, its shares of the odd
// site's self inverse and of the even site's self block into registers, the even
// site's hop rows into shared memory in the order in which they are read.
//
// Bound by latency: a step is a chain of some ten phases of a few thousand operations with a barrier each, so what
// counts is the length of every phase.  Row i of a site is formed by the eight lanes 8 i ... 8 i + 7, lane k from hop
// block k and an eighth of the self block (or inverse), and summed by shuffles that halve the values as they go:
// no partial rows in shared memory and no barrier for their sum.  FP32 products run on pairs of columns (two FMAs per
// instruction); in the resident variant a warp forms four rows, so that a value read from shared memory serves four.
// The rotations of the Hessenberg column are a chain of up to j complex operations by one warp; they are
// worked off by a warp of their own while the others form the odd half of the next step's product (which is in
// vain after the last step).  Cycles of a step before -> now: 56 dof on 16 CTAs, FP32: 25300 -> 23000; 16 dof on 8 CTAs,
// FP64: 52000 -> 32000, of which 9000 are the FP64 rate of the eight SMs.  One solve of the three-level cycle on
// 16^3x32 took 409 us on average and takes 370; of the two-level one on 8^4 in FP64 476 and 280.
#include <cooperative_groups.h>

#include "common.cuh"
#include "kernels.h"

namespace cg = cooperative_groups;

namespace {

constexpr int MAXM = 64;
constexpr int RES_NR = 56;   // largest coarse dof count of the resident variant (rows held in registers)

DD_HD size_t bidx(int site, int k, int n, int i, int j) { return (((size_t)site * 9 + k) * n + j) * n + i; }

// shared memory in units of cplx<T>, the same on host and device
struct Sizes {
  int xstride;   // gathered neighbour vectors: row stride (bank conflicts: eight rows are read at a time)
  int vstride;   // Krylov basis: row stride
  int rstride;   // dot-product partials: entries per dot
};
DD_HD Sizes sizes_of(int n, int len, int CL, bool resident) {
  Sizes z;
  z.xstride = resident ? RES_NR : n + 1;
  z.vstride = len;
  if (resident)
    while ((z.vstride & 7) != 4) ++z.vstride;
  z.rstride = CL == 16 ? CL + 4 : CL;
  return z;
}

template <typename T>
struct Smem {
  cplx<T>* Vb;     // [m+1][vstride] Krylov basis rows of the own even sites
  cplx<T>* xv;     // [ne_per*n] solution (even)
  cplx<T>* rv;     // [ne_per*n] residual / bhat
  cplx<T>* wv;     // [ne_per*n] new direction
  cplx<T>* be;     // [ne_per*n] b on the own even sites
  cplx<T>* bo;     // [no_per*n] b on the own odd sites
  cplx<T>* tv;     // [no_per*n] S_oo^{-1}(...) on the own odd sites
  cplx<T>* xs;     // [8][xstride] gathered neighbour vectors (resident: [8][quarter][7] pairs of columns (re, re, im, im))
  cplx<T>* us;     // [n]
  cplx<T>* wsum;   // [32] sums of the warps
  cplx<T>* red;    // [2][MAXM][rstride] partials of the dot products, then [rstride] of a norm
  cplx<T>* H;      // [m+1][m]
  cplx<T>* g;      // [m+1]
  cplx<T>* sn;     // [m]
  cplx<T>* y;      // [m]
  cplx<T>* hsum;   // [MAXM] reduced dots of the current pass; afterwards the running entry of the rotations
  cplx<T>* htot;   // [MAXM] sum of both CGS passes
  T* cs;           // [m]
  T* scal;         // [8] broadcast scalars inside the CTA
  uint4* eblk;     // resident: [2][7][nt] hop rows of the own even site per thread: two rows of a pair of columns
};

template <typename T>
DD_HD size_t smem_elems(int m, int nep, int nop, int n, int CL, const Sizes& z) {
  return (size_t)(m + 1) * z.vstride + 4 * (size_t)nep * n + 2 * (size_t)nop * n + 8 * (size_t)z.xstride + n + 32 +
         (size_t)(2 * MAXM + 1) * z.rstride + (size_t)(m + 1) * m + (m + 1) + 2 * (size_t)m + 2 * MAXM;
}

template <typename T>
__device__ Smem<T> carve(unsigned char* base, int m, int nep, int nop, int n, const Sizes& z) {
  // layout must match smem_elems()
  Smem<T> s;
  cplx<T>* p = reinterpret_cast<cplx<T>*>(base);
  s.xs = p; p += (size_t)8 * z.xstride;   // first: read 16 bytes at a time
  s.Vb = p; p += (size_t)(m + 1) * z.vstride;
  s.xv = p; p += (size_t)nep * n;
  s.rv = p; p += (size_t)nep * n;
  s.wv = p; p += (size_t)nep * n;
  s.be = p; p += (size_t)nep * n;
  s.bo = p; p += (size_t)nop * n;
  s.tv = p; p += (size_t)nop * n;
  s.us = p; p += (size_t)n;
  s.wsum = p; p += 32;
  s.red = p; p += (size_t)(2 * MAXM + 1) * z.rstride;
  s.H = p; p += (size_t)(m + 1) * m;
  s.g = p; p += (size_t)(m + 1);
  s.sn = p; p += (size_t)m;
  s.y = p; p += (size_t)m;
  s.hsum = p; p += (size_t)MAXM;
  s.htot = p; p += (size_t)MAXM;
  T* q = reinterpret_cast<T*>(p);
  s.cs = q; q += m;
  s.scal = q;
  q += 8;
  s.eblk = reinterpret_cast<uint4*>((reinterpret_cast<uintptr_t>(q) + 15) & ~uintptr_t(15));
  return s;
}

template <typename T>
struct Ctx {
  const cplx<T>* blk;
  const __half2* blkh;     // FP16 blocks (FP32 compute only) or null
  const float* bscale;     // per-site scale of blkh
  const cplx<T>* inv;
  const int* even;
  const int* odd;
  const int* nbr_e_of_o;   // [n_o][8] even-list index of neighbour k (k<4: +mu, k>=4: -mu)
  const int* nbr_o_of_e;   // [n_e][8]
  int n_e, n_o, nep, nop, n, CL, rank;
  int nw;                  // threads that form rows (the warp after them works off the rotations)
  int gk, gj;              // neighbour and component that this thread gathers
  int gx;                  // and where to (resident)
  int nbo, nbe;            // its neighbours' list indexes if a CTA has one site of each parity
  Sizes z;
};

// Operator rows held by one thread of the resident variant.  Warp w forms rows 4 w ... 4 w + 3 of a site; lane
// 4 k + q has a quarter of the columns of hop block k (up to 14, in pairs), and columns lane and lane + 32 of
// the self block and inverse.
constexpr int RP = RES_NR / 8;   // pairs of columns in a quarter
template <int NR>
struct RegRows {};
template <>
struct RegRows<RES_NR> {
  __half2 re[4][RP], im[4][RP];   // hop blocks of the odd site
  cplx<float> inv[4][2];          // the odd site's self inverse
  __half2 self[4][2];             // the even site's self block
  float so, se;                   // scales of the two sites' blocks
};

__device__ __forceinline__ void pack_cols(__half2 a, __half2 b, __half2& re, __half2& im) {
  re = __halves2half2(__low2half(a), __low2half(b));
  im = __halves2half2(__high2half(a), __high2half(b));
}
// acc (rr: re re, ii: im im, ri: the products of the imaginary part) += two columns of an FP16 row times x
__device__ __forceinline__ void cols_fma(float2& rr, float2& ii, float2& ri, __half2 mre, __half2 mim, float4 x) {
  const float2 a = __half22float2(mre), b = __half22float2(mim);
  const float2 xr = make_float2(x.x, x.y), xi = make_float2(x.z, x.w);
  rr = __ffma2_rn(a, xr, rr);
  ii = __ffma2_rn(b, xi, ii);
  ri = __ffma2_rn(a, xi, ri);
  ri = __ffma2_rn(b, xr, ri);
}
// v (re, im of four rows) = the lane's columns times x; get(rp, p, r0re, r0im, r1re, r1im) gives a pair of rows
template <class Get>
__device__ __forceinline__ void hop_rows(float* v, const float4* x, Get get) {
#pragma unroll
  for (int rp = 0; rp < 2; ++rp) {
    float2 rr0 = make_float2(0.f, 0.f), ii0 = rr0, ri0 = rr0, rr1 = rr0, ii1 = rr0, ri1 = rr0;
#pragma unroll
    for (int p = 0; p < RP; ++p) {
      __half2 a, b, c, d;
      get(rp, p, a, b, c, d);
      const float4 xp = x[p];
      cols_fma(rr0, ii0, ri0, a, b, xp);
      cols_fma(rr1, ii1, ri1, c, d, xp);
    }
    v[4 * rp] = (rr0.x + rr0.y) - (ii0.x + ii0.y);
    v[4 * rp + 1] = ri0.x + ri0.y;
    v[4 * rp + 2] = (rr1.x + rr1.y) - (ii1.x + ii1.y);
    v[4 * rp + 3] = ri1.x + ri1.y;
  }
}
// sum over the warp of eight values per lane: lane l returns value l / 4
__device__ __forceinline__ float fold_rows(float* v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int w = 4, off = 16; w >= 1; w >>= 1, off >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int k = 0; k < w; ++k) {
      const float keep = up ? v[k + w] : v[k], send = up ? v[k] : v[k + w];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// sum over the eight lanes of a group: lanes 0-3 return the real part, lanes 4-7 the imaginary part
template <typename T>
__device__ __forceinline__ T fold8(cplx<T> v) {
  const bool up = (threadIdx.x & 4) != 0;
  T r = (up ? v.im : v.re) + __shfl_xor_sync(0xffffffffu, up ? v.re : v.im, 4);
  r += __shfl_xor_sync(0xffffffffu, r, 2);
  return r + __shfl_xor_sync(0xffffffffu, r, 1);
}

// sum_j M(site, k)[i][j] x[j], j = j0, j0 + dj, ... from the compute-precision or the FP16 blocks
template <typename T>
__device__ __forceinline__ cplx<T> block_row(const Ctx<T>& cx, int site, int k, int i, const cplx<T>* x, int j0,
                                             int dj) {
  const int n = cx.n;
  // two accumulators: two independent chains of fused multiply-adds
  cplx<T> acc = czero<T>(), acc1 = czero<T>();
  int j = j0;
  if constexpr (sizeof(T) == 4) {
    if (cx.blkh) {
      const __half2* M = cx.blkh + bidx(site, k, n, i, 0);
#pragma unroll 4
      for (; j + dj < n; j += 2 * dj) {
        cfma(acc, ld_cplx(M, (size_t)j * n), x[j]);
        cfma(acc1, ld_cplx(M, (size_t)(j + dj) * n), x[j + dj]);
      }
      if (j < n) cfma(acc, ld_cplx(M, (size_t)j * n), x[j]);
      return T(cx.bscale[site]) * (acc + acc1);
    }
  }
  const cplx<T>* M = cx.blk + bidx(site, k, n, i, 0);
#pragma unroll 4
  for (; j + dj < n; j += 2 * dj) {
    cfma(acc, M[(size_t)j * n], x[j]);
    cfma(acc1, M[(size_t)(j + dj) * n], x[j + dj]);
  }
  if (j < n) cfma(acc, M[(size_t)j * n], x[j]);
  return acc + acc1;
}

// neighbour value (own gk, gj) of a site from its owner's array `src` into xs
template <typename T, int NR>
__device__ __forceinline__ void gather(const Ctx<T>& cx, const Smem<T>& s, cg::cluster_group& cluster, cplx<T>* src,
                                       int nb, int per) {
  const int q = per == 1 ? nb : nb / per;
  const cplx<T> v = cluster.map_shared_rank(src, q)[(nb - q * per) * cx.n + cx.gj];
  if constexpr (NR > 0) {
    T* d = reinterpret_cast<T*>(s.xs) + cx.gx;
    d[0] = v.re;
    d[2] = v.im;
  } else {
    s.xs[cx.gk * cx.z.xstride + cx.gj] = v;
  }
}

__device__ __forceinline__ void sync_rows(int nw) { asm volatile("bar.sync 1, %0;" ::"r"(nw) : "memory"); }

// t(own odd) = S^{-1} ( a*bo + c * sum_k D_k(o) v(even nbr_k) ), v read from the owners' array `src`; called by
// the first nw threads
template <typename T, int NR>
__device__ __forceinline__ void odd_phase(const Ctx<T>& cx, const Smem<T>& s, cg::cluster_group& cluster, cplx<T>* src,
                                          T a, T c, const RegRows<NR>& rows) {
  const int n = cx.n, t = threadIdx.x, i = t >> 3, k = t & 7;
  const bool act = t < 8 * n;
  if constexpr (NR > 0) {
    if (cx.rank >= cx.n_o) return;   // uniform in the CTA
    const int lane = t & 31, p = 8 * (t >> 5) + (lane >> 2);   // the scalar that this lane's fold returns
    if (c != T(0) && act) gather<T, NR>(cx, s, cluster, src, cx.nbo, 1);
    sync_rows(cx.nw);
    float u = 0.f;
    if (c != T(0)) {
      float v[8];
      hop_rows(v, reinterpret_cast<const float4*>(s.xs) + lane * RP,
               [&](int rp, int q, __half2& a0, __half2& b0, __half2& a1, __half2& b1) {
                 a0 = rows.re[2 * rp][q], b0 = rows.im[2 * rp][q];
                 a1 = rows.re[2 * rp + 1][q], b1 = rows.im[2 * rp + 1][q];
               });
      u = c * rows.so * fold_rows(v);
    }
    if ((lane & 3) == 0 && p < 2 * n) {
      if (a != T(0)) u += a * reinterpret_cast<const T*>(s.bo)[p];
      reinterpret_cast<T*>(s.us)[p] = u;
    }
    sync_rows(cx.nw);
    cplx<float> w[4] = {};
#pragma unroll
    for (int q = 0; q < 2; ++q)
      if (lane + 32 * q < n) {
        const cplx<float> uj = s.us[lane + 32 * q];
#pragma unroll
        for (int r = 0; r < 4; ++r) cfma(w[r], rows.inv[r][q], uj);
      }
    u = fold_rows(reinterpret_cast<float*>(w));
    if ((lane & 3) == 0 && p < 2 * n) reinterpret_cast<T*>(s.tv)[p] = u;
    return;
  }
  for (int so = 0; so < cx.nop; ++so) {
    const int o = cx.rank * cx.nop + so;
    if (o >= cx.n_o) break;   // uniform in the CTA
    const int site = cx.odd[o];
    if (c != T(0) && act)
      gather<T, NR>(cx, s, cluster, src, cx.nop == 1 && cx.nep == 1 ? cx.nbo : cx.nbr_e_of_o[o * 8 + cx.gk], cx.nep);
    sync_rows(cx.nw);
    cplx<T> acc = czero<T>();
    if (c != T(0) && act) {
      acc = c * block_row(cx, site, 1 + k, i, s.xs + k * cx.z.xstride, 0, 1);
    }
    T u = fold8(acc);
    if (act && (k & 3) == 0) {
      const int p = 2 * i + (k >> 2);
      if (a != T(0)) u += a * reinterpret_cast<const T*>(s.bo + so * n)[p];
      reinterpret_cast<T*>(s.us)[p] = u;
    }
    sync_rows(cx.nw);
    acc = czero<T>();
    if (act) {
      const cplx<T>* Mi = cx.inv + ((size_t)site * n) * n + i;
#pragma unroll 4
      for (int j = k; j < n; j += 8) cfma(acc, Mi[(size_t)j * n], s.us[j]);
    }
    u = fold8(acc);
    if (act && (k & 3) == 0) reinterpret_cast<T*>(s.tv + so * n)[2 * i + (k >> 2)] = u;
  }
}

// dst(own even) = a*be + sc * S(e) xloc(e) + c * sum_k D_k(e) t(odd nbr_k)  (t read from the owners' tv)
template <typename T, int NR>
__device__ __forceinline__ void even_phase(const Ctx<T>& cx, const Smem<T>& s, cg::cluster_group& cluster,
                                           const cplx<T>* xloc, cplx<T>* dst, T a, T sc, T c,
                                           const RegRows<NR>& rows) {
  const int n = cx.n, t = threadIdx.x, i = t >> 3, k = t & 7;
  const bool act = t < 8 * n;
  if constexpr (NR > 0) {
    if (cx.rank >= cx.n_e) return;   // uniform in the CTA
    const int lane = t & 31, p = 8 * (t >> 5) + (lane >> 2), nt = (8 * n + 31) & ~31;
    if (act) gather<T, NR>(cx, s, cluster, s.tv, cx.nbe, 1);
    __syncthreads();
    if (t < nt) {   // whole warps
      float v[8];
      const uint4* M = s.eblk + t;
      hop_rows(v, reinterpret_cast<const float4*>(s.xs) + lane * RP,
               [&](int rp, int q, __half2& a0, __half2& b0, __half2& a1, __half2& b1) {
                 const uint4 m = M[(rp * RP + q) * nt];
                 a0 = reinterpret_cast<const __half2&>(m.x), b0 = reinterpret_cast<const __half2&>(m.y);
                 a1 = reinterpret_cast<const __half2&>(m.z), b1 = reinterpret_cast<const __half2&>(m.w);
               });
#pragma unroll
      for (int r = 0; r < 8; ++r) v[r] *= c;
      if (sc != T(0))
#pragma unroll
        for (int q = 0; q < 2; ++q)
          if (lane + 32 * q < n) {
            const cplx<float> xj = sc * xloc[lane + 32 * q];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              const float2 f = __half22float2(rows.self[r][q]);
              cplx<float> w = cmk(v[2 * r], v[2 * r + 1]);
              cfma(w, cmk(f.x, f.y), xj);
              v[2 * r] = w.re;
              v[2 * r + 1] = w.im;
            }
          }
      float u = rows.se * fold_rows(v);
      if ((lane & 3) == 0 && p < 2 * n) {
        if (a != T(0)) u += a * reinterpret_cast<const T*>(s.be)[p];
        reinterpret_cast<T*>(dst)[p] = u;
      }
    }
    __syncthreads();
    return;
  }
  for (int se = 0; se < cx.nep; ++se) {
    const int e = cx.rank * cx.nep + se;
    if (e >= cx.n_e) break;
    const int site = cx.even[e];
    if (act)
      gather<T, NR>(cx, s, cluster, s.tv, cx.nop == 1 && cx.nep == 1 ? cx.nbe : cx.nbr_o_of_e[e * 8 + cx.gk], cx.nop);
    __syncthreads();
    cplx<T> acc = czero<T>();
    if (act) {
      acc = c * block_row(cx, site, 1 + k, i, s.xs + k * cx.z.xstride, 0, 1);
      if (sc != T(0)) acc = acc + sc * block_row(cx, site, 0, i, xloc + se * n, k, 8);
    }
    T v = fold8(acc);
    if (act && (k & 3) == 0) {
      const int p = 2 * i + (k >> 2);
      if (a != T(0)) v += a * reinterpret_cast<const T*>(s.be + se * n)[p];
      reinterpret_cast<T*>(dst + se * n)[p] = v;
    }
    __syncthreads();
  }
}

// h[d] = sum over all CTAs of conj(V_d) . w for d <= j and, with with_norm, h[j+1] = ||w||^2.
// Groups of 8 lanes own one d each and reduce with shuffles (fixed order); they then write the CTA's partial
// into every CTA's buffer `slot`, so after the barrier every CTA sums its own copy, four lanes per dot
// (identical in every CTA, local reads only).
template <typename T>
__device__ __forceinline__ void cluster_dots(const Ctx<T>& cx, const Smem<T>& s, cg::cluster_group& cluster,
                                             const cplx<T>* w, int j, int slot, int len, bool with_norm) {
  cplx<T>* red = s.red + (size_t)slot * MAXM * cx.z.rstride;
  const int grp = threadIdx.x >> 3, l = threadIdx.x & 7, ngrp = blockDim.x >> 3;
  const int dmax = with_norm ? j + 1 : j;
  for (int d0 = 0; d0 <= dmax; d0 += ngrp) {
    const int d = d0 + grp;
    cplx<T> acc = czero<T>();
    if (d <= j) {
      const cplx<T>* v = s.Vb + (size_t)d * cx.z.vstride;
      for (int e = l; e < len; e += 8) cdotc_acc(acc.re, acc.im, v[e], w[e]);
    } else if (d == dmax) {
      for (int e = l; e < len; e += 8) acc.re += cnorm2(w[e]);
    }
    const T r = fold8(acc), o = __shfl_xor_sync(0xffffffffu, r, 4);
    if (d <= dmax)
      for (int q = l; q < cx.CL; q += 8)
        cluster.map_shared_rank(red, q)[d * cx.z.rstride + cx.rank] = l < 4 ? cmk<T>(r, o) : cmk<T>(o, r);
  }
  cluster.sync();
  for (int d0 = 0; d0 <= dmax; d0 += (int)(blockDim.x >> 2)) {
    const int d = d0 + (int)(threadIdx.x >> 2);
    cplx<T> t = czero<T>();
    if (d <= dmax)
#pragma unroll 4
      for (int q = threadIdx.x & 3; q < cx.CL; q += 4) t = t + red[d * cx.z.rstride + q];
    // lanes 0, 1 of a quad: the real part, lanes 2, 3: the imaginary part
    const bool up = (threadIdx.x & 2) != 0;
    T r = (up ? t.im : t.re) + __shfl_xor_sync(0xffffffffu, up ? t.re : t.im, 2);
    r += __shfl_xor_sync(0xffffffffu, r, 1);
    if (d <= dmax && (threadIdx.x & 1) == 0) reinterpret_cast<T*>(s.hsum + d)[(threadIdx.x >> 1) & 1] = r;
  }
  __syncthreads();
}

// ||w||^2 over the cluster (rank-ordered; every CTA sums its own copy of the partials)
template <typename T>
__device__ T cluster_norm2(const Ctx<T>& cx, const Smem<T>& s, cg::cluster_group& cluster, const cplx<T>* w, int len) {
  cplx<T>* red = s.red + (size_t)2 * MAXM * cx.z.rstride;
  T a = T(0);
  for (int e = threadIdx.x; e < len; e += blockDim.x) a += cnorm2(w[e]);
  for (int off = 16; off >= 1; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
  if ((threadIdx.x & 31) == 0) s.wsum[threadIdx.x >> 5].re = a;
  __syncthreads();
  if (threadIdx.x < 32) {
    a = threadIdx.x < (blockDim.x >> 5) ? s.wsum[threadIdx.x].re : T(0);
    for (int off = 16; off >= 1; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
    if (threadIdx.x < cx.CL) cluster.map_shared_rank(red, threadIdx.x)[cx.rank] = cmk<T>(a, T(0));
  }
  cluster.sync();
  if (threadIdx.x == 0) {
    T t = T(0);
    for (int q = 0; q < cx.CL; ++q) t += red[q].re;
    s.scal[4] = t;
  }
  __syncthreads();
  return s.scal[4];
}

// dst += sign * sum_{d < k} c_d V_d: 8 lanes per element, each a strided share of d
// (the loop runs to a multiple of 32 so that whole warps take part in the shuffles)
template <typename T>
__device__ __forceinline__ void add_basis(const Ctx<T>& cx, const Smem<T>& s, cplx<T>* dst, const cplx<T>* c, int k,
                                          int len, T sign) {
  for (int t = threadIdx.x; t < ((8 * len + 31) & ~31); t += blockDim.x) {
    const int e = t >> 3;
    cplx<T> acc = czero<T>();
    if (e < len)
#pragma unroll 4
      for (int d = t & 7; d < k; d += 8) cfma(acc, c[d], s.Vb[(size_t)d * cx.z.vstride + e]);
    const T r = fold8(acc);
    if (e < len && (t & 3) == 0) reinterpret_cast<T*>(dst + e)[(t >> 2) & 1] += sign * r;
  }
}

// Column j of the Hessenberg matrix (htot, scal[6]) into R and g, by one warp: lane 0 carries the real part of the
// running entry through the earlier rotations and lane 1 the imaginary part; what does not depend on it is formed
// by all lanes before and after.  scal[2] = 1 if the cycle ends here.
template <typename T>
__device__ __forceinline__ void rotate_column(const Smem<T>& s, int j, int m, T target) {
  const int lane = threadIdx.x & 31;
  cplx<T>* cur = s.hsum;
  for (int i = lane; i < j; i += 32) cur[i + 1] = s.cs[i] * s.htot[i + 1];
  if (lane == 0) cur[0] = s.htot[0];
  __syncwarp();
  if (j > 0) {
    const int p = lane & 1;   // every lane computes; lanes 0 and 1 store
    T c = p ? cur[0].im : cur[0].re;
#pragma unroll 2
    for (int i = 0; i < j; ++i) {
      const cplx<T> si = s.sn[i];
      const T a = p ? cur[i + 1].im : cur[i + 1].re, im = p ? si.im : -si.im;
      const T o = __shfl_xor_sync(0xffffffffu, c, 1);
      c = a - si.re * c + im * o;   // cs h_{i+1} - conj(sn) h_i
      __syncwarp();
      if (lane < 2) reinterpret_cast<T*>(cur + i + 1)[p] = c;
    }
  }
  __syncwarp();
  for (int i = lane; i < j; i += 32) s.H[(size_t)i * m + j] = s.cs[i] * cur[i] + s.sn[i] * s.htot[i + 1];
  if (lane == 0) {
    // |sn| = hn / rr, so |g_{j+1}| follows from |g_j| (scal[7]); one root and one inverse each for |h_j| and rr
    const T hn = s.scal[6];
    const cplx<T> h = cur[j], gj = s.g[j];
    const T n2 = cnorm2(h), aa = sqrt(n2), rr = sqrt(n2 + hn * hn);
    T c = T(1), f = T(0);
    cplx<T> sg = czero<T>();
    if (rr != T(0)) {
      const T ir = T(1) / rr;
      f = hn * ir;
      c = aa * ir;
      sg = aa == T(0) ? cmk<T>(T(1), T(0)) : (f * (T(1) / aa)) * h;
      if (aa == T(0)) f = T(1);
    }
    s.cs[j] = c;
    s.sn[j] = sg;
    s.H[(size_t)j * m + j] = c * h + hn * sg;
    s.g[j + 1] = T(-1) * (cconj(sg) * gj);
    s.g[j] = c * gj;
    const T est = f * s.scal[7];
    s.scal[7] = est;
    s.scal[2] = est <= target || hn == T(0) || j + 1 == m ? T(1) : T(0);
  }
  __syncwarp();
}

template <typename T, int NR>
__global__ void __launch_bounds__(512, 1) k_coarsest_cluster(Ctx<T> cx0, const cplx<T>* __restrict__ b, cplx<T>* __restrict__ x, size_t rstride,
                                   int m, int max_cycles, double tol, int* iters) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cg::cluster_group cluster = cg::this_cluster();
  Ctx<T> cx = cx0;
  cx.rank = (int)cluster.block_rank();
  cx.nw = (int)blockDim.x - 32;
  const int n = cx.n;
  const int len = cx.nep * n;
  cx.z = sizes_of(n, len, cx.CL, NR > 0);
  Smem<T> s = carve<T>(smem_raw, m, cx.nep, cx.nop, n, cx.z);
  const cplx<T>* pb = b + (size_t)blockIdx.y * rstride;
  cplx<T>* px = x + (size_t)blockIdx.y * rstride;
  const bool forms_rows = (int)threadIdx.x < cx.nw;   // the last warp works off the rotations meanwhile
  cx.gk = threadIdx.x / n;
  cx.gj = threadIdx.x - cx.gk * n;
  cx.nbo = cx.gk < 8 && cx.rank < cx.n_o ? cx.nbr_e_of_o[cx.rank * 8 + cx.gk] : 0;   // used with nep = nop = 1
  cx.nbe = cx.gk < 8 && cx.rank < cx.n_e ? cx.nbr_o_of_e[cx.rank * 8 + cx.gk] : 0;
  RegRows<NR> rows;
  if constexpr (NR > 0) {
    const int t = threadIdx.x, lane = t & 31, i0 = 4 * (t >> 5), k = lane >> 2, nt = (8 * n + 31) & ~31;
    const int pq = (n + 7) / 8, j0 = 2 * pq * (lane & 3);   // pairs in a quarter of the columns, the lane's first column
    const bool ho = t < nt && cx.rank < cx.n_o, he = t < nt && cx.rank < cx.n_e;
    const int so = ho ? cx.odd[cx.rank] : 0, se = he ? cx.even[cx.rank] : 0;
    rows.so = ho ? cx.bscale[so] : 0.f;
    rows.se = he ? cx.bscale[se] : 0.f;
    // rows i0 ... i0 + 3 of column j
    auto load = [&](const __half2* M, bool in, int j, __half2* r) {
      if (in && (n & 3) == 0) {
        const uint4 v = *reinterpret_cast<const uint4*>(M + (size_t)j * n + i0);
        r[0] = reinterpret_cast<const __half2&>(v.x), r[1] = reinterpret_cast<const __half2&>(v.y);
        r[2] = reinterpret_cast<const __half2&>(v.z), r[3] = reinterpret_cast<const __half2&>(v.w);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) r[q] = in && i0 + q < n ? M[(size_t)j * n + i0 + q] : __half2();
      }
    };
    const __half2 *Mo = cx.blkh + bidx(so, 1 + k, n, 0, 0), *Me = cx.blkh + bidx(se, 1 + k, n, 0, 0);
#pragma unroll
    for (int p = 0; p < RP; ++p) {
      const int j = j0 + 2 * p;   // n is even
      __half2 a[4], c[4];
      load(Mo, ho && p < pq && j < n, j, a);
      load(Mo, ho && p < pq && j < n, j + 1, c);
#pragma unroll
      for (int r = 0; r < 4; ++r) pack_cols(a[r], c[r], rows.re[r][p], rows.im[r][p]);
      load(Me, he && p < pq && j < n, j, a);
      load(Me, he && p < pq && j < n, j + 1, c);
      if (t < nt)
#pragma unroll
        for (int rp = 0; rp < 2; ++rp) {
          __half2 m[4];
          pack_cols(a[2 * rp], c[2 * rp], m[0], m[1]);
          pack_cols(a[2 * rp + 1], c[2 * rp + 1], m[2], m[3]);
          s.eblk[(rp * RP + p) * nt + t] =
              make_uint4(reinterpret_cast<const unsigned&>(m[0]), reinterpret_cast<const unsigned&>(m[1]),
                         reinterpret_cast<const unsigned&>(m[2]), reinterpret_cast<const unsigned&>(m[3]));
        }
    }
    const __half2* Ms = cx.blkh + bidx(se, 0, n, 0, 0);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int j = lane + 32 * q;
      __half2 a[4];
      load(Ms, he && j < n, j, a);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        rows.self[r][q] = a[r];
        rows.inv[r][q] = ho && j < n && i0 + r < n ? cx.inv[((size_t)so * n + j) * n + i0 + r] : czero<float>();
      }
    }
    // columns beyond n of the gathered vectors stay zero
    for (int e = t; e < 8 * RES_NR; e += blockDim.x) s.xs[e] = czero<T>();
    const int q = cx.gj / (2 * pq), w = cx.gj - 2 * pq * q;
    cx.gx = ((4 * cx.gk + q) * RP + (w >> 1)) * 4 + (w & 1);
  }
  // own b, zero x
  for (int t = threadIdx.x; t < len; t += blockDim.x) {
    const int e = cx.rank * cx.nep + t / n;
    s.be[t] = e < cx.n_e ? pb[(size_t)cx.even[e] * n + t % n] : czero<T>();
    s.xv[t] = s.rv[t] = s.wv[t] = czero<T>();
  }
  for (int t = threadIdx.x; t < cx.nop * n; t += blockDim.x) {
    const int o = cx.rank * cx.nop + t / n;
    s.bo[t] = o < cx.n_o ? pb[(size_t)cx.odd[o] * n + t % n] : czero<T>();
  }
  __syncthreads();
  // bhat_e = b_e - D_eo S_oo^{-1} b_o  -> rv
  if (forms_rows) odd_phase<T, NR>(cx, s, cluster, s.xv, T(1), T(0), rows);
  cluster.sync();
  even_phase<T, NR>(cx, s, cluster, s.xv, s.rv, T(1), T(0), T(-1), rows);
  const T bnorm = sqrt(cluster_norm2<T>(cx, s, cluster, s.rv, len));
  const T target = (T)tol * bnorm;
  // keep bhat: be <- rv (be is not needed any more)
  for (int t = threadIdx.x; t < len; t += blockDim.x) s.be[t] = s.rv[t];
  __syncthreads();
  T beta = bnorm;
  int total = 0;
  for (int cycle = 0; cycle < max_cycles; ++cycle) {
    if (!(beta > target)) break;   // converged (or zero rhs): uniform in the cluster
    const T iv = T(1) / beta;
    for (int t = threadIdx.x; t < len; t += blockDim.x) s.Vb[t] = iv * s.rv[t];
    for (int k = threadIdx.x; k <= m; k += blockDim.x) s.g[k] = k ? czero<T>() : cmk<T>(beta, T(0));
    if (threadIdx.x == 0) s.scal[7] = beta;
    cluster.sync();
    int kk = 0;
    for (int j = 0; j < m; ++j) {
      cplx<T>* vj = s.Vb + (size_t)j * cx.z.vstride;
      // w = Dhat v_j, and the rotations of the previous step
      if (forms_rows) odd_phase<T, NR>(cx, s, cluster, vj, T(0), T(1), rows);
      else if (j > 0) rotate_column(s, j - 1, m, target);
      cluster.sync();
      if (j > 0 && s.scal[2] != T(0)) break;   // the same in every CTA
      even_phase<T, NR>(cx, s, cluster, vj, s.wv, T(0), T(1), T(-1), rows);
      // CGS2; the second pass also sums ||w'||^2, and ||w''||^2 = ||w'||^2 - sum_d |h2_d|^2
      // (w'' = w' - V h2 with h2 = V^+ w' and V orthonormal), which saves a reduction
      for (int pass = 0; pass < 2; ++pass) {
        cluster_dots<T>(cx, s, cluster, s.wv, j, pass, len, pass == 1);
        if (!forms_rows) {
          const int lane = threadIdx.x & 31;
          for (int d = lane; d <= j; d += 32) s.htot[d] = pass == 0 ? s.hsum[d] : s.htot[d] + s.hsum[d];
          if (pass == 1) {   // ||w''||^2 (strided partials, shuffle tree) and the inverse of its root
            T h2 = T(0);
            for (int d = lane; d <= j; d += 32) h2 += cnorm2(s.hsum[d]);
            for (int off = 16; off >= 1; off >>= 1) h2 += __shfl_xor_sync(0xffffffffu, h2, off);
            const T w2 = s.hsum[j + 1].re - h2, hn = sqrt(w2 > T(0) ? w2 : T(0));
            if (lane == 0) {
              s.scal[6] = hn;
              s.scal[3] = hn > T(0) ? T(1) / hn : T(0);
            }
          }
        }
        add_basis(cx, s, s.wv, s.hsum, j + 1, len, T(-1));   // w -= sum_d h_d V_d
        __syncthreads();
      }
      kk = j + 1;
      if (kk < m) {
        const T ivn = s.scal[3];
        cplx<T>* vn = vj + cx.z.vstride;
        for (int e = threadIdx.x; e < len; e += blockDim.x) vn[e] = ivn * s.wv[e];
        cluster.sync();
      }
    }
    if (kk == m && !forms_rows) rotate_column(s, m - 1, m, target);
    total += kk;
    // y = R^{-1} g: with y_i known, all lanes of a warp subtract its column from the rows above
    __syncthreads();
    if (threadIdx.x < 32) {
      for (int i = threadIdx.x; i < kk; i += 32) {   // the diagonal's inverse in its place
        cplx<T>& d = s.H[(size_t)i * m + i];
        const T dn = cnorm2(d);
        d = dn > T(0) ? (T(1) / dn) * cconj(d) : czero<T>();
      }
      __syncwarp();
      for (int i = kk - 1; i >= 0; --i) {
        const cplx<T> yi = s.g[i] * s.H[(size_t)i * m + i];
        for (int l = threadIdx.x; l < i; l += 32) s.g[l] = s.g[l] - s.H[(size_t)l * m + i] * yi;
        if (threadIdx.x == 0) s.y[i] = yi;
        __syncwarp();
      }
    }
    __syncthreads();
    add_basis(cx, s, s.xv, s.y, kk, len, T(1));   // x += V y
    cluster.sync();
    if (cycle + 1 == max_cycles) break;
    // true residual r = bhat - Dhat x
    if (forms_rows) odd_phase<T, NR>(cx, s, cluster, s.xv, T(0), T(1), rows);
    cluster.sync();
    even_phase<T, NR>(cx, s, cluster, s.xv, s.rv, T(1), T(-1), T(1), rows);   // uses be = bhat as b
    beta = sqrt(cluster_norm2<T>(cx, s, cluster, s.rv, len));
  }
  // z_o = S_oo^{-1} (b_o - D_oe x_e); write x
  cluster.sync();
  if (forms_rows) odd_phase<T, NR>(cx, s, cluster, s.xv, T(1), T(-1), rows);
  __syncthreads();
  for (int t = threadIdx.x; t < len; t += blockDim.x) {
    const int e = cx.rank * cx.nep + t / n;
    if (e < cx.n_e) px[(size_t)cx.even[e] * n + t % n] = s.xv[t];
  }
  for (int t = threadIdx.x; t < cx.nop * n; t += blockDim.x) {
    const int o = cx.rank * cx.nop + t / n;
    if (o < cx.n_o) px[(size_t)cx.odd[o] * n + t % n] = s.tv[t];
  }
  if (cx.rank == 0 && threadIdx.x == 0 && iters) atomicAdd(iters, total);
  cluster.sync();   // no CTA exits while others may still read its shared memory
}

template <typename T>
size_t smem_bytes(int m, int nep, int nop, int n, int CL, bool resident) {
  size_t b = smem_elems<T>(m, nep, nop, n, CL, sizes_of(n, nep * n, CL, resident)) * sizeof(cplx<T>) + (m + 8) * sizeof(T) + 16;
  if (resident) b += (size_t)2 * RP * ((8 * n + 31) & ~31) * sizeof(uint4);
  return b + 64;
}

}  // namespace

namespace dd {

// the dynamic shared-memory limit is a process-wide attribute of the kernel: raised to the device
// maximum, so that hierarchies set up later with a smaller coarsest level do not lower it
template <typename T, int NR>
bool cluster_fits(int CL, int threads, size_t sm) {
  if (cudaFuncSetAttribute(k_coarsest_cluster<T, NR>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) !=
      cudaSuccess) {
    cudaGetLastError();
    cudaFuncSetAttribute(k_coarsest_cluster<T, NR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  }
  if (CL > 8) cudaFuncSetAttribute(k_coarsest_cluster<T, NR>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CL;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(CL, 1, 1);
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = sm;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int nclusters = 0;
  if (cudaOccupancyMaxActiveClusters(&nclusters, k_coarsest_cluster<T, NR>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return nclusters >= 1;
}

// Chooses the cluster size (16 if the device can co-schedule it, else 8, 4, 2)
// and reports whether the cluster kernel can run this level (shared memory).
// For FP32 it also records whether the resident variant (FP16 blocks, one even
// and one odd site per CTA) fits.
template <typename T>
int coarsest_cluster_plan(const CoarsestPlanIn& in, CoarsestPlan* plan) {
  const int n_e = in.n_even, n_o = in.n_odd;
  for (int CL : {16, 8, 4, 2}) {
    if (CL > n_e || CL > n_o) continue;
    const int nep = (n_e + CL - 1) / CL, nop = (n_o + CL - 1) / CL;
    const size_t sm = smem_bytes<T>(in.m, nep, nop, in.n, CL, false);
    if (sm > 220 * 1024) continue;
    if (in.n > RES_NR) return 0;   // eight threads form a row, at most 480 a site (512 keep 128 registers each)
    int threads = ((8 * in.n + 31) / 32) * 32;
    if (threads < 256) threads = 256;
    threads += 32;   // the warp that works off the rotations
    if (!cluster_fits<T, 0>(CL, threads, sm)) continue;
    plan->CL = CL;
    plan->nep = nep;
    plan->nop = nop;
    plan->threads = threads;
    plan->smem = sm;
    plan->res_nr = 0;
    plan->res_smem = 0;
    if constexpr (sizeof(T) == 4) {
      const size_t smr = smem_bytes<T>(in.m, nep, nop, in.n, CL, true);
      if (nep == 1 && nop == 1 && in.n <= RES_NR && threads <= 512 && smr <= 227 * 1024 &&
          cluster_fits<T, RES_NR>(CL, threads, smr)) {
        plan->res_nr = RES_NR;
        plan->res_smem = smr;
      }
    }
    return 1;
  }
  return 0;
}

template <typename T>
cudaError_t coarsest_cluster_solve(cplx<T>* x, const cplx<T>* b, const CoarseOp<T>& op, const CoarsestPlan& plan,
                                   const CoarsestGeo& geo, int nrhs, size_t rstride, int m, int max_cycles, double tol,
                                   int* iters, cudaStream_t st) {
  Ctx<T> cx;
  cx.blk = op.blk;
  cx.blkh = op.blkh;
  cx.bscale = op.bscale;
  cx.inv = op.selfinv;
  cx.even = geo.even;
  cx.odd = geo.odd;
  cx.nbr_e_of_o = geo.nbr_e_of_o;
  cx.nbr_o_of_e = geo.nbr_o_of_e;
  cx.n_e = geo.n_even;
  cx.n_o = geo.n_odd;
  cx.nep = plan.nep;
  cx.nop = plan.nop;
  cx.n = op.n;
  cx.CL = plan.CL;
  cx.rank = 0;
  const bool resident = sizeof(T) == 4 && op.blkh && plan.res_nr > 0;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = plan.CL;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(plan.CL, nrhs, 1);
  cfg.blockDim = dim3(plan.threads, 1, 1);
  cfg.dynamicSmemBytes = resident ? plan.res_smem : plan.smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  count_launch();
  if constexpr (sizeof(T) == 4)
    if (resident)
      return cudaLaunchKernelEx(&cfg, k_coarsest_cluster<T, RES_NR>, cx, b, x, rstride, m, max_cycles, tol, iters);
  return cudaLaunchKernelEx(&cfg, k_coarsest_cluster<T, 0>, cx, b, x, rstride, m, max_cycles, tol, iters);
}

#define INST(T)                                                                                                     \
  template int coarsest_cluster_plan<T>(const CoarsestPlanIn&, CoarsestPlan*);                                      \
  template cudaError_t coarsest_cluster_solve<T>(cplx<T>*, const cplx<T>*, const CoarseOp<T>&, const CoarsestPlan&,  \
                                                 const CoarsestGeo&, int, size_t, int, int, double, int*, cudaStream_t);
INST(float)
INST(double)
#undef INST

}  // namespace dd
