// Coarse-level kernels: the Galerkin operators D_{l+1} = P_l^+ D_l P_l are
// nearest-neighbour stencils of dense n x n complex blocks (Sec. 1, Sec. 2):
//   (D phi)(A) = S(A) phi(A) + sum_mu [ F_mu(A) phi(A + mu) + B_mu(A) phi(A - mu) ].
// Blocks are stored column-major per (site, k) with k = 0 self, 1..4 forward,
// 5..8 backward, so that the threads computing consecutive rows of one site
// read consecutive words.
#include <atomic>

#include <cooperative_groups.h>

#include "common.cuh"
#include "kernels.h"
#include "tma.cuh"

namespace cg = cooperative_groups;

namespace {

DD_HD size_t bidx(int site, int k, int n, int i, int j) { return (((size_t)site * 9 + k) * n + j) * n + i; }

template <typename T>
__device__ void cta_sum3(T& a, T& b, T& c, T* sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  for (int off = 16; off >= 1; off >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, off);
    b += __shfl_xor_sync(0xffffffffu, b, off);
    c += __shfl_xor_sync(0xffffffffu, c, off);
  }
  if (lane == 0) { sh[3 * warp] = a; sh[3 * warp + 1] = b; sh[3 * warp + 2] = c; }
  __syncthreads();
  a = b = c = T(0);
  for (int w = 0; w < nw; ++w) { a += sh[3 * w]; b += sh[3 * w + 1]; c += sh[3 * w + 2]; }
  __syncthreads();
}

// (D phi)(A): one CTA per coarse site, one thread per (row i, block k); the
// neighbour vectors are staged in shared memory and the 9 partial rows are
// summed in shared memory.  Blocks are column-major, so the threads of one k
// read consecutive words for every column j.
template <typename T, bool RESID, typename BS>
__global__ void k_coarse_apply(cplx<T>* __restrict__ out, const cplx<T>* __restrict__ in,
                               const cplx<T>* __restrict__ bsrc, const BS* __restrict__ blk,
                               const float* __restrict__ bscale, Geom g, int n, size_t rstride, int sel, int sel_mu,
                               int in_chir) {
  extern __shared__ unsigned char smem_raw[];
  cplx<T>* xs = reinterpret_cast<cplx<T>*>(smem_raw);   // [9][n] neighbour vectors
  cplx<T>* part = xs + 9 * n;                           // [9][n] partial rows
  __shared__ int nbr[9];
  __shared__ int take[9];
  const int site = blockIdx.x;
  const size_t ro = (size_t)blockIdx.y * rstride;
  const cplx<T>* pin = in + ro;
  if (threadIdx.x < 9) {
    int c[4];
    geom_coords(g, site, c);
    const int k = threadIdx.x;
    int nb = site;
    bool tk = sel == SEL_FULL || sel == SEL_AGG_SELF;
    if (k > 0) {
      const int mu = (k - 1) % 4, dir = k <= 4 ? +1 : -1;
      nb = geom_neighbor(g, c, mu, dir);
      const bool internal = hop_internal(g, c, mu, dir, g.fA);
      if (sel == SEL_FULL) tk = true;
      else if (sel == SEL_AGG_SELF) tk = internal;
      else if (sel == SEL_AGG_FWD) tk = dir > 0 && mu == sel_mu && !internal;
      else tk = dir < 0 && mu == sel_mu && !internal;
    }
    nbr[k] = nb;
    take[k] = tk;
  }
  __syncthreads();
  // the term of a hop that leaves the aggregate: sites without it are not written (nor read by the product with P^+)
  if ((sel == SEL_AGG_FWD && !take[1 + sel_mu]) || (sel == SEL_AGG_BWD && !take[5 + sel_mu])) return;
  const int h = n / 2;
  for (int e = threadIdx.x; e < 9 * n; e += blockDim.x) {
    const int k = e / n, j = e % n;
    const bool keep = take[k] && (in_chir < 0 || (j < h) == (in_chir == 0));
    xs[e] = keep ? pin[(size_t)nbr[k] * n + j] : czero<T>();
  }
  __syncthreads();
  const int k = threadIdx.x / n, i = threadIdx.x % n;
  if (k < 9) {
    cplx<T> acc = czero<T>();
    if (take[k]) {
      const BS* M = blk + (((size_t)site * 9 + k) * n) * n + i;
      const cplx<T>* x = xs + k * n;
#pragma unroll 8
      for (int j = 0; j < n; ++j) cfma(acc, ld_cplx(M, (size_t)j * n), x[j]);
      if (bscale) acc = T(bscale[site]) * acc;
    }
    part[k * n + i] = acc;
  }
  __syncthreads();
  if (threadIdx.x < n) {
    cplx<T> y = czero<T>();
#pragma unroll
    for (int q = 0; q < 9; ++q) y = y + part[q * n + threadIdx.x];
    const size_t a = ro + (size_t)site * n + threadIdx.x;
    out[a] = RESID ? bsrc[a] - y : y;
  }
}

// Even-odd pieces of the coarsest solve (Sec. 3: odd-even preconditioned GMRES),
// with D = [[S_ee, D_eo], [D_oe, S_oo]] and the self blocks S inverted at setup.
// k_schur_odd: on every odd site A,  t(A) = S(A)^{-1} ( a*b(A) + c*(D_oe x)(A) )
//              (even entries of t are not written)
// k_schur_even: on every even site A, y(A) = a*b(A) + s*S(A) x(A) + c*(D_eo t)(A);
//              odd entries of y are set to zero.
template <typename T, typename BS>
__global__ void k_schur_odd(cplx<T>* __restrict__ t, const cplx<T>* __restrict__ x, const cplx<T>* __restrict__ b,
                            const BS* __restrict__ blk, const float* __restrict__ bscale,
                            const cplx<T>* __restrict__ inv,
                            const int* __restrict__ odd_sites, Geom g, int n, size_t rstride, double a, double c) {
  extern __shared__ unsigned char smem_raw[];
  cplx<T>* xs = reinterpret_cast<cplx<T>*>(smem_raw);   // [8][n]
  cplx<T>* part = xs + 8 * n;                           // [8][n]
  cplx<T>* u = part + 8 * n;                            // [n]
  __shared__ int nbr[8];
  const size_t ro = (size_t)blockIdx.y * rstride;
  const int site = odd_sites[blockIdx.x];
  if (threadIdx.x < 8) {
    int cc[4];
    geom_coords(g, site, cc);
    const int k = threadIdx.x;
    nbr[k] = geom_neighbor(g, cc, k % 4, k < 4 ? +1 : -1);
  }
  __syncthreads();
  if (x && c != 0.0)
    for (int e = threadIdx.x; e < 8 * n; e += blockDim.x) xs[e] = x[ro + (size_t)nbr[e / n] * n + e % n];
  __syncthreads();
  const int k = threadIdx.x / n, i = threadIdx.x % n;
  if (k < 8) {
    cplx<T> acc = czero<T>();
    if (x && c != 0.0) {
      const BS* M = blk + (((size_t)site * 9 + 1 + k) * n) * n + i;
      const cplx<T>* xv = xs + k * n;
#pragma unroll 8
      for (int j = 0; j < n; ++j) cfma(acc, ld_cplx(M, (size_t)j * n), xv[j]);
      if (bscale) acc = T(bscale[site]) * acc;
    }
    part[k * n + i] = acc;
  }
  __syncthreads();
  if (threadIdx.x < n) {
    cplx<T> y = czero<T>();
#pragma unroll
    for (int q = 0; q < 8; ++q) y = y + part[q * n + threadIdx.x];
    y = T(c) * y;
    if (b && a != 0.0) y = y + T(a) * b[ro + (size_t)site * n + threadIdx.x];
    u[threadIdx.x] = y;
  }
  __syncthreads();
  if (threadIdx.x < n) {
    cplx<T> acc = czero<T>();
    const cplx<T>* Mi = inv + ((size_t)site * n) * n + threadIdx.x;
#pragma unroll 8
    for (int j = 0; j < n; ++j) cfma(acc, Mi[(size_t)j * n], u[j]);
    t[ro + (size_t)site * n + threadIdx.x] = acc;
  }
}

template <typename T, typename BS>
__global__ void k_schur_even(cplx<T>* __restrict__ y, const cplx<T>* __restrict__ x, const cplx<T>* __restrict__ t,
                             const cplx<T>* __restrict__ b, const BS* __restrict__ blk,
                             const float* __restrict__ bscale, Geom g, int n, size_t rstride, double a, double s,
                             double c) {
  extern __shared__ unsigned char smem_raw[];
  cplx<T>* xs = reinterpret_cast<cplx<T>*>(smem_raw);   // [9][n]
  cplx<T>* part = xs + 9 * n;                           // [9][n]
  __shared__ int nbr[9];
  const int site = blockIdx.x;
  const size_t ro = (size_t)blockIdx.y * rstride;
  int cc[4];
  geom_coords(g, site, cc);
  if (geom_parity(cc) != 0) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) y[ro + (size_t)site * n + i] = czero<T>();
    return;
  }
  if (threadIdx.x < 9) {
    const int k = threadIdx.x;
    nbr[k] = k == 0 ? site : geom_neighbor(g, cc, (k - 1) % 4, k <= 4 ? +1 : -1);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < 9 * n; e += blockDim.x) {
    const int k = e / n, j = e % n;
    const cplx<T>* src = k == 0 ? x : t;
    const double w = k == 0 ? s : c;
    xs[e] = (src && w != 0.0) ? src[ro + (size_t)nbr[k] * n + j] : czero<T>();
  }
  __syncthreads();
  const int k = threadIdx.x / n, i = threadIdx.x % n;
  if (k < 9) {
    cplx<T> acc = czero<T>();
    const double w = k == 0 ? s : c;
    if (w != 0.0 && (k == 0 ? x : t)) {
      const BS* M = blk + (((size_t)site * 9 + k) * n) * n + i;
      const cplx<T>* xv = xs + k * n;
#pragma unroll 8
      for (int j = 0; j < n; ++j) cfma(acc, ld_cplx(M, (size_t)j * n), xv[j]);
      if (bscale) acc = T(bscale[site]) * acc;
    }
    part[k * n + i] = T(w) * acc;
  }
  __syncthreads();
  if (threadIdx.x < n) {
    cplx<T> v = czero<T>();
#pragma unroll
    for (int q = 0; q < 9; ++q) v = v + part[q * n + threadIdx.x];
    const size_t o = ro + (size_t)site * n + threadIdx.x;
    if (b && a != 0.0) v = v + T(a) * b[o];
    y[o] = v;
  }
}

// One colour sweep of SAP on a coarse level: one CTA per SAP block; thread t owns
// the rows t, t + blockDim.x, ... (at most RPT) of the block, row = (site, i) in
// block-local order (bsite / bloc tables).  rho = (b - D z)_B, k MR steps on D_B
// (hops leaving the block dropped), z_B += e_B; the operator is read from global
// memory.
// Largest CTA per rows-per-thread variant: what coarse_sap_sweep may launch, so that the compiler keeps the registers
// within it (blocks of up to 3072 rows in FP64 and 3840 in FP32).
template <typename T, int RPT> constexpr int coarse_sap_threads() {
  return sizeof(T) == 8 ? (RPT == 1 ? 896 : RPT == 4 ? 576 : 384) : (RPT == 1 ? 1024 : RPT == 4 ? 800 : 480);
}
template <typename T, typename BS, int RPT>
__global__ void __launch_bounds__(coarse_sap_threads<T, RPT>()) k_coarse_sap(cplx<T>* __restrict__ z, const cplx<T>* __restrict__ bsrc,
                             const BS* __restrict__ blk, const float* __restrict__ bscale, Geom g, int n,
                             size_t rstride, const int* __restrict__ blocks, int k_mr,
                             const int* __restrict__ bsite, const int* __restrict__ bloc) {
  extern __shared__ unsigned char smem_raw[];
  cplx<T>* rs = reinterpret_cast<cplx<T>*>(smem_raw);        // [vB * n]
  T* sh = reinterpret_cast<T*>(rs + (size_t)g.vB * n);          // [warps][3]
  const int b = blocks[blockIdx.x];
  const int rows = g.vB * n;
  const int* bs = bsite + (size_t)b * g.vB;
  const size_t ro = (size_t)blockIdx.y * rstride;
  cplx<T>* pz = z + ro;
  cplx<T> r[RPT], xs[RPT], p[RPT];
#pragma unroll
  for (int q = 0; q < RPT; ++q) {
    r[q] = czero<T>();
    xs[q] = czero<T>();
    const int row = threadIdx.x + q * blockDim.x;
    if (row < rows) {
      const int loc = row / n, i = row - loc * n;
      const int site = bs[loc];
      int c[4];
      geom_coords(g, site, c);
      cplx<T> acc = czero<T>();
      // self block, then the forward (1 + mu) and backward (5 + mu) blocks; written as
      // explicit direction loops (a single 9-way loop over k was mis-executed here)
      {
        const cplx<T>* v = pz + (size_t)site * n;
        for (int j = 0; j < n; ++j) cfma(acc, ld_cplx(blk, bidx(site, 0, n, i, j)), v[j]);
      }
      for (int mu = 0; mu < 4; ++mu)
        for (int sd = 0; sd < 2; ++sd) {
          const int dir = sd ? -1 : +1, k = sd ? 5 + mu : 1 + mu;
          const cplx<T>* v = pz + (size_t)geom_neighbor(g, c, mu, dir) * n;
          for (int j = 0; j < n; ++j) cfma(acc, ld_cplx(blk, bidx(site, k, n, i, j)), v[j]);
        }
      const T sc = bscale ? T(bscale[site]) : T(1);
      r[q] = bsrc[ro + (size_t)site * n + i] - sc * acc;
    }
  }
  for (int it = 0; it < k_mr; ++it) {
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
      const int row = threadIdx.x + q * blockDim.x;
      if (row < rows) rs[row] = r[q];
    }
    __syncthreads();
    T nre = T(0), nim = T(0), den = T(0);
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
      p[q] = czero<T>();
      const int row = threadIdx.x + q * blockDim.x;
      if (row < rows) {
        const int loc = row / n, i = row - loc * n;
        const int site = bs[loc];
        int c[4];
        geom_coords(g, site, c);
        cplx<T> acc = czero<T>();
        {
          const cplx<T>* v = rs + (size_t)loc * n;
#pragma unroll 8
          for (int j = 0; j < n; ++j) cfma(acc, ld_cplx(blk, bidx(site, 0, n, i, j)), v[j]);
        }
        for (int mu = 0; mu < 4; ++mu)
          for (int sd = 0; sd < 2; ++sd) {
            const int dir = sd ? -1 : +1, k = sd ? 5 + mu : 1 + mu;
            if (!hop_internal(g, c, mu, dir, g.fB)) continue;
            const cplx<T>* v = rs + (size_t)bloc[geom_neighbor(g, c, mu, dir)] * n;
#pragma unroll 8
            for (int j = 0; j < n; ++j) cfma(acc, ld_cplx(blk, bidx(site, k, n, i, j)), v[j]);
          }
        const T sc = bscale ? T(bscale[site]) : T(1);
        p[q] = sc * acc;
        const cplx<T> tt = cdotc(p[q], r[q]);
        nre += tt.re;
        nim += tt.im;
        den += cnorm2(p[q]);
      }
    }
    cta_sum3(nre, nim, den, sh);
    const cplx<T> alpha = den > T(0) ? cmk<T>(nre / den, nim / den) : czero<T>();
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
      cfma(xs[q], alpha, r[q]);
      r[q] = r[q] - alpha * p[q];
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < RPT; ++q) {
    const int row = threadIdx.x + q * blockDim.x;
    if (row < rows) {
      const int loc = row / n, i = row - loc * n;
      const size_t a = ro + (size_t)bs[loc] * n + i;
      z[a] = z[a] + xs[q];
    }
  }
}

// shared-memory layout of k_coarse_sap_cluster (byte offsets, 16-byte aligned)
struct SapSmem {
  size_t rfull, pbuf, part, red, sh, slot, bar, total;
};
DD_HD size_t al16(size_t x) { return (x + 15) & ~size_t(15); }
DD_HD SapSmem sap_smem_layout(int vB, int n, int spc, int nsl, size_t ts) {
  SapSmem L;
  size_t o = al16((size_t)spc * nsl * n * n * 2 * ts);
  L.rfull = o;
  o = al16(o + (size_t)vB * n * 2 * ts);
  L.pbuf = o;
  o = al16(o + (size_t)2 * vB * n * 2 * ts);
  L.part = o;
  o = al16(o + (size_t)9 * spc * n * 2 * ts);
  L.red = o;
  o = al16(o + (size_t)2 * 16 * 4 * ts);
  L.sh = o;
  o = al16(o + (size_t)(32 * 3 + 4) * ts);
  L.slot = o;
  o = al16(o + (size_t)spc * 9 * sizeof(int));
  L.bar = o;
  L.total = al16(o + 8);
  return L;
}

// SAP colour sweep on a coarse level with one thread-block cluster per SAP
// block.  CTA q of the cluster owns `spc` sites of the block, one thread per
// (row, block k) of its sites.  The blocks of its sites that couple inside the
// SAP block (self block included) are staged once into shared memory by bulk
// copies; the hops leaving the block are only needed for rho = b - D z and are
// read from global memory.  Every CTA keeps the whole block residual r and the
// whole MR direction p = D_B r in shared memory: after computing p on its own
// rows a CTA writes them, with its partial dot products, into every CTA of the
// cluster (distributed shared memory), so each MR step needs one cluster
// barrier; p and the partials are double-buffered across steps.  The partial
// dot products are summed in rank order, so every CTA computes the same alpha
// and applies r <- r - alpha p to its whole copy.  Same arithmetic as
// k_coarse_sap: rho = (b - D z)_B, k MR steps on D_B, z_B += e_B.
template <typename T>
__global__ void __launch_bounds__(768, 2) k_coarse_sap_cluster(cplx<T>* __restrict__ z, const cplx<T>* __restrict__ bsrc,
                                     const cplx<T>* __restrict__ blk, Geom g, int n,
                                     size_t rstride, int nrhs, const int* __restrict__ blocks, int k_mr, int spc,
                                     int nsl, int* err, const int* __restrict__ bsite,
                                     const int* __restrict__ bloc) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  // the next sweep (launched with programmatic stream serialization) may stage its blocks while
  // this one runs; it waits for this grid before reading z or b
  pdl_launch_dependents();
  cg::cluster_group cluster = cg::this_cluster();
  const int CLS = (int)cluster.num_blocks();
  const int rank = (int)cluster.block_rank();
  const int vB = g.vB;
  const int b = blocks[blockIdx.x / CLS];
  const int rows = spc * n;
  const size_t nn = (size_t)n * n;
  const SapSmem L = sap_smem_layout(vB, n, spc, nsl, sizeof(T));
  cplx<T>* stage = reinterpret_cast<cplx<T>*>(smem_raw);                      // [spc][nsl][n][n]
  cplx<T>* rfull = reinterpret_cast<cplx<T>*>(smem_raw + L.rfull);            // [vB*n]
  cplx<T>* pbuf = reinterpret_cast<cplx<T>*>(smem_raw + L.pbuf);              // [2][vB*n]
  cplx<T>* part = reinterpret_cast<cplx<T>*>(smem_raw + L.part);              // [9][rows]
  T* red = reinterpret_cast<T*>(smem_raw + L.red);                            // [2][16][4]
  T* sh = reinterpret_cast<T*>(smem_raw + L.sh);                              // [32][3] + 3
  int* slot = reinterpret_cast<int*>(smem_raw + L.slot);                      // [spc][9]
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(smem_raw + L.bar);
  const int* own = bsite + (size_t)b * vB + rank * spc;   // own sites, block-local order
  // slot of block k of own site sl in the staged array (-1: the hop leaves the SAP block)
  if (threadIdx.x < spc) {
    int c[4];
    geom_coords(g, own[threadIdx.x], c);
    // slots in k order (self, forward mu = 0..3, backward mu = 0..3), explicit direction loops
    int* sl9 = slot + threadIdx.x * 9;
    int ns = 0;
    sl9[0] = ns++;
    for (int sd = 0; sd < 2; ++sd)
      for (int mu = 0; mu < 4; ++mu)
        sl9[(sd ? 5 : 1) + mu] = hop_internal(g, c, mu, sd ? -1 : +1, g.fB) ? ns++ : -1;
  }
  if (threadIdx.x == 0) mbar_init(bar, 1);
  __syncthreads();
  if (threadIdx.x < 32) {
    int cnt = 0;
    for (int e = 0; e < spc * 9; ++e) cnt += slot[e] >= 0 ? 1 : 0;
    if (threadIdx.x == 0) mbar_arrive_expect_tx(bar, (unsigned)(cnt * nn * sizeof(cplx<T>)));
    __syncwarp();
    for (int e = threadIdx.x; e < spc * 9; e += 32) {
      const int sl = e / 9, k = e % 9, q = slot[e];
      if (q >= 0)
        bulk_g2s(stage + ((size_t)sl * nsl + q) * nn, blk + ((size_t)own[sl] * 9 + k) * nn,
                 (unsigned)(nn * sizeof(cplx<T>)), bar);
    }
  }
  const int k = threadIdx.x / rows;
  const int rl = threadIdx.x - k * rows;
  const int sl = rl / n, i = rl - (rl / n) * n;
  const int site = own[sl];
  int q = -1, nb = site, nloc = 0;
  if (k < 9) {
    q = slot[sl * 9 + k];
    if (k > 0) {
      int c[4];
      geom_coords(g, site, c);
      nb = geom_neighbor(g, c, (k - 1) % 4, k <= 4 ? +1 : -1);
    }
    nloc = q >= 0 ? bloc[nb] : 0;
  }
  const cplx<T>* Ms = stage + ((size_t)sl * nsl + (q >= 0 ? q : 0)) * nn + i;   // staged row i (column-major)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  int ok = 1;
  pdl_wait();   // the previous kernel's z and b are complete from here on
  // the right-hand sides of the batch one after the other, on the blocks staged once
  for (int rh = 0; rh < nrhs; ++rh) {
    const size_t ro = (size_t)rh * rstride;
    // rho = b - D z on the own rows: hops leaving the block from global memory ...
    cplx<T> acc = czero<T>();
    if (k < 9 && q < 0) {
      const cplx<T>* M = blk + ((size_t)site * 9 + k) * nn + i;
      const cplx<T>* v = z + ro + (size_t)nb * n;
#pragma unroll 8
      for (int j = 0; j < n; ++j) cfma(acc, M[(size_t)j * n], v[j]);
    }
    if (rh == 0) {
      ok = __syncthreads_and(mbar_wait_bounded(bar, 0) ? 1 : 0);
      if (!ok && threadIdx.x == 0) atomicExch(err, 2);
    }
    // ... and the blocks inside it from shared memory
    if (k < 9 && q >= 0) {
      const cplx<T>* v = z + ro + (size_t)nb * n;
#pragma unroll 8
      for (int j = 0; j < n; ++j) cfma(acc, Ms[(size_t)j * n], v[j]);
    }
    if (k < 9) part[k * rows + rl] = acc;
    __syncthreads();
    cplx<T> r = czero<T>(), xs = czero<T>();
    if (threadIdx.x < rows) {
      cplx<T> d = czero<T>();
#pragma unroll
      for (int m = 0; m < 9; ++m) d = d + part[m * rows + threadIdx.x];
      r = bsrc[ro + (size_t)own[threadIdx.x / n] * n + threadIdx.x % n] - d;
      for (int c = 0; c < CLS; ++c) cluster.map_shared_rank(rfull, c)[(size_t)rank * rows + threadIdx.x] = r;
    }
    cluster.sync();
    for (int it = 0; it < k_mr; ++it) {
      const int buf = it & 1;
      cplx<T>* pb = pbuf + (size_t)buf * vB * n;
      T* rb = red + buf * 64;
      // p = D_B r on the own rows, from the staged blocks and the local copy of r
      if (k < 9) {
        cplx<T> a = czero<T>();
        if (q >= 0) {
          const cplx<T>* v = rfull + (size_t)nloc * n;
#pragma unroll 8
          for (int j = 0; j < n; ++j) cfma(a, Ms[(size_t)j * n], v[j]);
        }
        part[k * rows + rl] = a;
      }
      __syncthreads();
      cplx<T> p = czero<T>();
      T nre = T(0), nim = T(0), den = T(0);
      if (threadIdx.x < rows) {
#pragma unroll
        for (int m = 0; m < 9; ++m) p = p + part[m * rows + threadIdx.x];
        const cplx<T> t = cdotc(p, r);
        nre = t.re;
        nim = t.im;
        den = cnorm2(p);
        for (int c = 0; c < CLS; ++c) cluster.map_shared_rank(pb, c)[(size_t)rank * rows + threadIdx.x] = p;
      }
      for (int off = 16; off >= 1; off >>= 1) {
        nre += __shfl_xor_sync(0xffffffffu, nre, off);
        nim += __shfl_xor_sync(0xffffffffu, nim, off);
        den += __shfl_xor_sync(0xffffffffu, den, off);
      }
      if (lane == 0) { sh[3 * warp] = nre; sh[3 * warp + 1] = nim; sh[3 * warp + 2] = den; }
      __syncthreads();
      if (warp == 0) {   // warp partials summed by a shuffle tree (fixed order), then sent to every CTA
        T a = lane < nw ? sh[3 * lane] : T(0);
        T bb = lane < nw ? sh[3 * lane + 1] : T(0);
        T cc = lane < nw ? sh[3 * lane + 2] : T(0);
        for (int off = 16; off >= 1; off >>= 1) {
          a += __shfl_xor_sync(0xffffffffu, a, off);
          bb += __shfl_xor_sync(0xffffffffu, bb, off);
          cc += __shfl_xor_sync(0xffffffffu, cc, off);
        }
        if (lane < CLS) {
          T* dst = cluster.map_shared_rank(rb, lane) + rank * 4;
          dst[0] = a;
          dst[1] = bb;
          dst[2] = cc;
        }
      }
      cluster.sync();
      T a = T(0), bb = T(0), cc = T(0);
      for (int c = 0; c < CLS; ++c) { a += rb[c * 4]; bb += rb[c * 4 + 1]; cc += rb[c * 4 + 2]; }
      const cplx<T> alpha = cc > T(0) ? cmk<T>(a / cc, bb / cc) : czero<T>();
      if (threadIdx.x < rows) {
        cfma(xs, alpha, r);
        r = r - alpha * p;
      }
      for (int e = threadIdx.x; e < vB * n; e += blockDim.x) rfull[e] = rfull[e] - alpha * pb[e];
      __syncthreads();
    }
    if (ok && threadIdx.x < rows) {
      const size_t a = ro + (size_t)own[threadIdx.x / n] * n + threadIdx.x % n;
      z[a] = z[a] + xs;
    }
    // every CTA is done with its copies of r, p and the partials before the next right-hand side
    // writes into them
    if (rh + 1 < nrhs) cluster.sync();
  }
  if (!ok && threadIdx.x == 0) mbar_wait_bounded(bar, 0);   // no copy may still be in flight at exit
}

// ---------------------------------------------------------------------------
// Coarse SAP on FP16 blocks (FP32 compute): one thread-block cluster per SAP block as above.  A warp forms RPL rows of a
// site, its lanes each every 32nd column of the site's concatenated blocks, RB right-hand sides at a time (a block
// entry is read and widened once for them, and they share the barriers).
//
// What bounds it is the chain of one MR step, about 2.5 us: matrix-vector product, exchange, sums, update.  So a column
// of RPL rows is one load of the blocks and one of the vector for 4 RPL RB FMAs; the lanes share the sums out as they
// fold them; a CTA keeps r on its own sites and their neighbours in the SAP block only, so p goes to the few CTAs that
// own those, and the CTAs' partial dot products to all, by asynchronous stores that complete on the target's
// mbarrier (a cluster barrier in their place waits for every store to be acknowledged: 25 against 31 us per
// sweep).  The blocks inside the SAP block are staged before the launch waits for the previous sweep, first in
// slot order, so that an MR step runs through one contiguous matrix; the others are read from L2 for rho.
// ddamg_smooth on level 1 of 16^3x32 (4^3x8 sites, 40 dof, 2^4 blocks), 10 sweeps of 4 MR steps: 252 us for one
// right-hand side and 1590 for twelve, where one thread per (row, block), partial rows through shared memory
// and cluster barriers took 342 and 3103.

// z in L2 only (values written by other CTAs of the launch)
__device__ __forceinline__ cplx<float> ldz(const cplx<float>* p) {
  const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
  return cmk<float>(v.x, v.y);
}

struct SapHSmem {
  size_t zn, rf, pf, xa, zs, part, nbr, kof, nin, sc, voff, uoff, nu, pairs, np, flag, bar, total;
};
// A pair (own site of a CTA, CTA of the cluster) in 16 bits.  The exchanged vectors alone, 16 vB n bytes, keep a SAP
// block below 7264 sites at n = 2, so a CTA of two or more has less than 4096 (and vB n below 2^15, as the positions
// in r need, which are kept in shorts).
constexpr int SAPH_SITES = 4096;   // most sites of a CTA
DD_HD unsigned short saph_pair(int sl, int cta) { return (unsigned short)(sl << 4 | cta); }
DD_HD int saph_pair_site(unsigned short p) { return p >> 4; }
DD_HD int saph_pair_cta(unsigned short p) { return p & 15; }
// nstage: staged blocks of the CTA; nblk: SAP blocks whose tables it keeps
DD_HD SapHSmem saph_smem_layout(int vB, int n, int spc, int RB, int nstage, int nblk) {
  SapHSmem L;
  const size_t cs = sizeof(cplx<float>);
  size_t o = al16((size_t)nstage * n * n * sizeof(__half2));
  // the neighbours' z are read for rho only, which r takes the place of
  L.zn = L.rf = o;
  o = al16(o + (size_t)RB * n * cs * (9 * spc > vB ? 9 * spc : vB));
  L.pf = o;
  o = al16(o + (size_t)2 * RB * vB * n * cs);
  L.xa = o;
  o = al16(o + (size_t)RB * spc * n * cs);
  L.zs = o;
  o = al16(o + (size_t)RB * spc * n * cs);
  L.part = o;  // [2][16][RB] dot products of the CTAs
  o = al16(o + (size_t)2 * 16 * RB * sizeof(float4));
  L.nbr = o;   // [nblk][spc][9] sites by slot
  o = al16(o + (size_t)nblk * spc * 9 * sizeof(int));
  L.kof = o;   // [nblk][spc][9] block index k of a slot
  o = al16(o + (size_t)nblk * spc * 9 * sizeof(int));
  L.nin = o;   // [nblk][spc] slots inside the SAP block
  o = al16(o + (size_t)nblk * spc * sizeof(int));
  L.sc = o;    // [nblk][spc] scales of the sites' blocks
  o = al16(o + (size_t)nblk * spc * sizeof(float));
  L.voff = o;  // [nblk][spc][9 n] position in r of a column inside the SAP block
  o = al16(o + (size_t)nblk * spc * 9 * n * sizeof(short));
  L.uoff = o;  // [nblk][9 spc] sites whose r the CTA keeps (positions in the SAP block): its own, then neighbours
  o = al16(o + (size_t)nblk * 9 * spc * sizeof(short));
  L.nu = o;    // [nblk] their number
  o = al16(o + (size_t)nblk * sizeof(int));
  L.pairs = o;   // [nblk][16 spc] (own site, other CTA that owns a neighbour of it)
  o = al16(o + (size_t)nblk * spc * 16 * sizeof(short));
  L.np = o;      // [nblk] their number
  o = al16(o + (size_t)nblk * sizeof(int));
  L.flag = o;
  o = al16(o + 16);
  L.bar = o;   // staged blocks; exchange buffers 0, 1
  L.total = al16(o + 24);
  return L;
}
constexpr int SAPH_W = 14;   // most warps
// warps for `rows` rows of a CTA in groups of rpl: the fewest that share them out as evenly as SAPH_W
DD_HD int saph_warps(int rows, int rpl) {
  const int groups = rows / rpl, per = (groups + SAPH_W - 1) / SAPH_W;
  return (groups + per - 1) / per;
}
// rows of a warp (n is even).  Eight rows: two lanes per column with four rows each, so that the eight lanes of a
// 16-byte load hit all banks at an odd multiple of eight dofs (lanes of 32 different columns: half of them)
DD_HD int saph_rpl(int n) { return n % 8 == 0 ? 8 : n % 4 == 0 ? 4 : 2; }

// tables of SAP block q of the CTA (own: its spc sites there): slots in k order, those inside the SAP block first.  A
// barrier follows.
__device__ __forceinline__ void saph_tables(const Geom& g, int n, int RB, const int* own, int spc, const int* bloc,
                                            const float* bscale, unsigned char* smem, const SapHSmem& L, int q) {
  int* nbr = reinterpret_cast<int*>(smem + L.nbr) + q * spc * 9;
  int* kof = reinterpret_cast<int*>(smem + L.kof) + q * spc * 9;
  int* nin = reinterpret_cast<int*>(smem + L.nin) + q * spc;
  short* voff = reinterpret_cast<short*>(smem + L.voff) + (size_t)q * spc * 9 * n;
  // one lane per (site, k): whether its hop stays inside, then its slot by the ranks of the inside ones
  for (int sl = threadIdx.x >> 5; sl < spc; sl += blockDim.x >> 5) {
    const int k = threadIdx.x & 31;
    int nb = own[sl], loc = -1;
    if (k < 9) {
      bool in = true;
      if (k > 0) {
        int c[4];
        geom_coords(g, nb, c);
        const int mu = (k - 1) & 3, dir = k <= 4 ? +1 : -1;
        in = hop_internal(g, c, mu, dir, g.fB);
        nb = geom_neighbor(g, c, mu, dir);
      }
      if (in) loc = bloc[nb];
    }
    const unsigned m = __ballot_sync(0xffffffffu, k < 9 && loc >= 0);
    const int ins = __popc(m), before = __popc(m & ((1u << k) - 1));
    if (k == 0) {
      nin[sl] = ins;
      reinterpret_cast<float*>(smem + L.sc)[q * spc + sl] = bscale[own[sl]];
    }
    if (k < 9) {
      const int slot = loc >= 0 ? before : ins + k - before;
      nbr[sl * 9 + slot] = nb;
      kof[sl * 9 + slot] = k;
    }
    for (int s = 0; s < ins; ++s) {   // the lane of slot s is the s-th that is inside
      const int at = __shfl_sync(0xffffffffu, loc, __fns(m, 0, s + 1)) * n * RB;
      for (int j = k; j < n; j += 32) voff[(sl * 9 + s) * n + j] = (short)(at + j);
    }
  }
}

// by one thread, a barrier after saph_tables and one before saph_block's exchanges: the sites whose r the CTA keeps (its
// own, then every other site that one of them has inside the block, once) and the CTAs its sites go to
__device__ __forceinline__ void saph_links(int n, int RB, int spc, int rank, unsigned char* smem, const SapHSmem& L, int q) {
  const int* nin = reinterpret_cast<const int*>(smem + L.nin) + q * spc;
  const short* voff = reinterpret_cast<const short*>(smem + L.voff) + (size_t)q * spc * 9 * n;
  short* u = reinterpret_cast<short*>(smem + L.uoff) + q * 9 * spc;
  unsigned short* pairs = reinterpret_cast<unsigned short*>(smem + L.pairs) + q * spc * 16;
  int cnt = 0, np = 0;
  for (int sl = 0; sl < spc; ++sl) u[cnt++] = (short)(rank * spc + sl);
  for (int sl = 0; sl < spc; ++sl) {
    unsigned to = 1u << rank;
    for (int m = 1; m < nin[sl]; ++m) {
      const int loc = voff[(sl * 9 + m) * n] / (n * RB);
      bool seen = false;
      for (int e = 0; e < cnt; ++e) seen = seen || u[e] == loc;
      if (!seen) u[cnt++] = (short)loc;
      const int t = loc / spc;
      if (!(to >> t & 1u)) pairs[np++] = saph_pair(sl, t);
      to |= 1u << t;
    }
  }
  reinterpret_cast<int*>(smem + L.nu)[q] = cnt;
  reinterpret_cast<int*>(smem + L.np)[q] = np;
}

// v[0 .. NV) summed over the lanes of the warp that are equal modulo M (1 or 2), which share the values out as they fold
// them: lane l returns value (l / M) / (32 / M / NV)
template <int NV, int M>
__device__ __forceinline__ float warp_fold(float (&v)[NV], int lane) {
  int off = 16;
#pragma unroll
  for (int w = NV / 2; w >= 1; w >>= 1, off >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int k = 0; k < w; ++k) {
      const float keep = up ? v[k + w] : v[k], send = up ? v[k] : v[k + w];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
  for (; off >= M; off >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
  return v[0];
}

// RPL neighbouring rows of a column
template <int RPL>
struct HalfRows {
  unsigned w[RPL];
  __device__ __forceinline__ void load(const __half2* p) {
    if constexpr (RPL == 2) {
      *reinterpret_cast<uint2*>(w) = *reinterpret_cast<const uint2*>(p);
    } else {
#pragma unroll
      for (int r = 0; r < RPL; r += 4) {
        const uint4 v = *reinterpret_cast<const uint4*>(p + r);
        w[r] = v.x;
        w[r + 1] = v.y;
        w[r + 2] = v.z;
        w[r + 3] = v.w;
      }
    }
  }
};

// One SAP block (table q of the CTA), right-hand sides rh0 .. rh0 + nb - 1 (nb <= RB): rho = (b - D z)_B, k MR steps,
// z_B += e_B.  seq: exchanges of the CTA so far (their parity picks the buffer).  stage: [spc][nst slots][n][n] in
// shared memory (every slot inside the SAP block is staged); ext(sl, slot): a block that is not; staged(): a barrier
// that waits for the staged blocks; false: they did not arrive, z is not written.
template <int RB, int RPL, bool L2Z, class Ext, class Staged>
__device__ __forceinline__ void saph_block(cg::cluster_group& cluster, cplx<float>* z, const cplx<float>* bsrc,
                                           int vB, int n, FDiv fn, size_t rstride, int rh0, int nb, int k_mr,
                                           int spc, const int* own, unsigned char* smem, const SapHSmem& L, int q, unsigned& seq,
                                           int* err, const __half2* stage, int nst, Ext ext, Staged staged) {
  using C = cplx<float>;
  constexpr int M = RPL == 8 ? 2 : 1, RL = RPL / M;   // lanes per column, rows of a lane
  using HR = HalfRows<RL>;
  constexpr int NV = 2 * RL * RB;                     // sums of a lane's rows: [right-hand side][row][re, im]
  C* zn = reinterpret_cast<C*>(smem + L.zn);             // [RB][spc][9 n] z of the own sites and neighbours (rho)
  // vectors on the SAP block, [vB][RB][n]; only the own sites and their neighbours in the block are kept up to date
  C* rf = reinterpret_cast<C*>(smem + L.rf);             // residual
  C* pf = reinterpret_cast<C*>(smem + L.pf);             // [2] exchanged vectors: r, then p
  unsigned long long* xbar = reinterpret_cast<unsigned long long*>(smem + L.bar) + 1;   // [2]
  C* xa = reinterpret_cast<C*>(smem + L.xa);             // [RB][rows] correction of the own rows
  C* zs = reinterpret_cast<C*>(smem + L.zs);             // [RB][rows] z of the own rows
  float4* part = reinterpret_cast<float4*>(smem + L.part);   // [2][16][RB]
  const short* us = reinterpret_cast<const short*>(smem + L.uoff) + q * 9 * spc;
  const int* nbr = reinterpret_cast<const int*>(smem + L.nbr) + q * spc * 9;
  const int* nin = reinterpret_cast<const int*>(smem + L.nin) + q * spc;
  const float* sc = reinterpret_cast<const float*>(smem + L.sc) + q * spc;
  const short* voff = reinterpret_cast<const short*>(smem + L.voff) + (size_t)q * spc * 9 * n;
  const int CLS = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nth >> 5;
  const int rows = spc * n, N = vB * n, nn = n * n, zst = spc * 9 * n;
  for (int e0 = tid; e0 < RB * zst; e0 += 4 * nth) {   // four loads in flight per thread
    C v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = e0 + u * nth, t = fdiv(e, fn), rr = RB == 1 ? 0 : t / (9 * spc);
      v[u] = czero<float>();
      if (e < RB * zst && rr < nb) {
        const C* pz = z + (size_t)(rh0 + rr) * rstride + (size_t)nbr[t - rr * 9 * spc] * n + (e - t * n);
        v[u] = L2Z ? ldz(pz) : *pz;
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (e0 + u * nth < RB * zst) zn[e0 + u * nth] = v[u];
  }
  bool ok = staged();
  const int nu = reinterpret_cast<const int*>(smem + L.nu)[q];
  const int npair = reinterpret_cast<const int*>(smem + L.np)[q];
  const unsigned short* pairs = reinterpret_cast<const unsigned short*>(smem + L.pairs) + q * spc * 16;
  // acc += column `h` of RPL rows times v
  auto column = [&](float (&acc)[NV], const HR& h, const C (&v)[RB]) {
#pragma unroll
    for (int r = 0; r < RL; ++r) {
      const float2 m = __half22float2(*reinterpret_cast<const __half2*>(&h.w[r]));
#pragma unroll
      for (int rr = 0; rr < RB; ++rr) {
        float& re = acc[(rr * RL + r) * 2];
        float& im = acc[(rr * RL + r) * 2 + 1];
        re = fmaf(m.x, v[rr].re, re);
        re = fmaf(-m.y, v[rr].im, re);
        im = fmaf(m.x, v[rr].im, im);
        im = fmaf(m.y, v[rr].re, im);
      }
    }
  };
  // lane -> (right-hand side, row of the group, re / im) of the value it holds after the fold
  constexpr int LPV = 32 / M / NV;
  const int vi = lane / M / LPV, v_rr = vi / (2 * RL), v_row = lane % M * RL + vi / 2 % RL, v_c = vi & 1;
  const bool v_on = lane / M % LPV == 0;
  const int c0 = lane / M, r0 = lane % M * RL;   // first column and row of the lane
  // The own sites of d (an exchange buffer) to the CTAs that own their neighbours in the block, whose sites come back
  // (adjacency is symmetric), a warp's asynchronous stores per site and CTA; and with dots the own rows' <d, r>, |d|^2 to every CTA.
  // Everything completes on the target's barrier, so that nobody waits for more than the data.  A buffer is free again
  // two exchanges later: a CTA sends the next vector but one only after every CTA's next dot products have come.
  auto exchange = [&](C* d, bool dots) {
    const unsigned buf = seq & 1, parity = (seq >> 1) & 1;
    ++seq;
    __syncthreads();
    if (tid == 0)
      mbar_arrive_expect_tx(&xbar[buf], (unsigned)((nu - spc) * RB * n * sizeof(C) + CLS * RB * sizeof(float4)));
    for (int p = warp; p < npair; p += nw) {
      const int sl = saph_pair_site(pairs[p]), t = saph_pair_cta(pairs[p]);
      float4* o = reinterpret_cast<float4*>(d + (size_t)(rank * spc + sl) * RB * n);
      for (int e = lane; e < RB * n / 2; e += 32) st_async_cluster(o + e, o[e], &xbar[buf], t);
    }
    for (int rr = nw > 1 ? warp - 1 : 0; rr >= 0 && rr < RB; rr += nw > 1 ? nw - 1 : 1) {   // a warp per right-hand side
      float v[4] = {0.f, 0.f, 0.f, 0.f};
      if (dots)
        for (int e = lane; e < rows; e += 32) {
          const int so = e / n, o = ((rank * spc + so) * RB + rr) * n + (e - so * n);
          cdotc_acc(v[0], v[1], d[o], rf[o]);
          cnorm2_acc(v[2], d[o]);
        }
#pragma unroll
      for (int k = 0; k < 3; ++k)
        for (int off = 16; off >= 1; off >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], off);
      if (lane < CLS)
        st_async_cluster(&part[(buf * 16 + rank) * RB + rr], make_float4(v[0], v[1], v[2], 0.f), &xbar[buf], lane);
    }
    if (!mbar_wait_bounded(&xbar[buf], parity)) {
      ok = false;
      atomicExch(err, 2);
    }
    return (const float4*)part + buf * 16 * RB;
  };
  auto buffer = [&] { return pf + (size_t)(seq & 1) * RB * N; };
  C* px = buffer();
  for (int g0 = warp; g0 < rows / RPL; g0 += nw) {
    const int row0 = g0 * RPL, sl = row0 / n, i0 = row0 - sl * n;
    float acc[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) acc[k] = 0.f;
    const C* vz = zn + sl * 9 * n;
    const __half2* A = stage + sl * nst * nn + i0 + r0;
    int c = c0;
#pragma unroll 4
    for (; c < nst * n; c += 32 / M) {
      C v[RB];
#pragma unroll
      for (int rr = 0; rr < RB; ++rr) v[rr] = vz[rr * zst + c];
      HR h;
      h.load(A + c * n);
      column(acc, h, v);
    }
#pragma unroll 5
    for (; c < 9 * n; c += 32 / M) {
      const int slot = c / n;
      HR h;
      h.load(ext(sl, slot) + (c - slot * n) * n + i0 + r0);
      C v[RB];
#pragma unroll
      for (int rr = 0; rr < RB; ++rr) v[rr] = vz[rr * zst + c];
      column(acc, h, v);
    }
    const float s = warp_fold<NV, M>(acc, lane);
    if (v_on) {
      const int i = i0 + v_row, row = row0 + v_row;
      const float b = v_rr < nb ? reinterpret_cast<const float*>(bsrc + (size_t)(rh0 + v_rr) * rstride +
                                                                 (size_t)own[sl] * n + i)[v_c] : 0.f;
      reinterpret_cast<float*>(px + ((rank * spc + sl) * RB + v_rr) * n + i)[v_c] = b - sc[sl] * s;
      reinterpret_cast<float*>(zs + v_rr * rows + row)[v_c] =
          reinterpret_cast<const float*>(vz + v_rr * zst + i)[v_c];                       // slot 0 is the site itself
    }
  }
  for (int e = tid; e < RB * rows; e += nth) xa[e] = czero<float>();
  exchange(px, false);
  for (int t = warp; t < nu * RB; t += nw) {   // r at the kept sites; every warp is past rho (the exchange's barrier)
    const int at = (us[t / RB] * RB + t % RB) * n;
    for (int j = lane; j < n; j += 32) rf[at + j] = px[at + j];
  }
  __syncthreads();
  for (int it = 0; it < k_mr; ++it) {
    C* pb = buffer();
    for (int g0 = warp; g0 < rows / RPL; g0 += nw) {
      const int row0 = g0 * RPL, sl = row0 / n, i0 = row0 - sl * n;
      float acc[NV];
#pragma unroll
      for (int k = 0; k < NV; ++k) acc[k] = 0.f;
      const short* vo = voff + sl * 9 * n;
      const int nc = nin[sl] * n;
      const __half2* A = stage + sl * nst * nn + i0 + r0;
#pragma unroll 4
      for (int c = c0; c < nc; c += 32 / M) {
        const int o = vo[c];
        C v[RB];
#pragma unroll
        for (int rr = 0; rr < RB; ++rr) v[rr] = rf[rr * n + o];
        HR h;
        h.load(A + c * n);
        column(acc, h, v);
      }
      const float s = warp_fold<NV, M>(acc, lane);
      if (v_on)
        reinterpret_cast<float*>(pb + ((rank * spc + sl) * RB + v_rr) * n + i0 + v_row)[v_c] = sc[sl] * s;
    }
    const float4* dp = exchange(pb, true);
    // alpha from the CTAs' partial sums in rank order (the same in every CTA), then r on the kept sites
    C alpha[RB];
#pragma unroll
    for (int rr = 0; rr < RB; ++rr) {
      float re = 0.f, im = 0.f, den = 0.f;
#pragma unroll
      for (int c = 0; c < 16; ++c)
        if (c < CLS) {
          const float4 t = dp[c * RB + rr];
          re += t.x;
          im += t.y;
          den += t.z;
        }
      alpha[rr] = den > 0.f ? cmk<float>(re / den, im / den) : czero<float>();
    }
    for (int t = warp; t < nu * RB; t += nw) {
      const int s = t / RB, rr = t - s * RB, at = (us[s] * RB + rr) * n;
      C al = alpha[0];
#pragma unroll
      for (int k = 1; k < RB; ++k)
        if (rr == k) al = alpha[k];
      for (int j = lane; j < n; j += 32) {
        const C r = rf[at + j];
        if (s < spc) cfma(xa[rr * rows + s * n + j], al, r);
        rf[at + j] = r - al * pb[at + j];
      }
    }
    __syncthreads();
  }
  if (__syncthreads_and(ok ? 1 : 0))   // and before the next right-hand sides' z take the place of r
    for (int e = tid; e < nb * rows; e += nth) {
      const int rr = e / rows, o = e - rr * rows, so = o / n;
      z[(size_t)(rh0 + rr) * rstride + (size_t)own[so] * n + (o - so * n)] = zs[e] + xa[e];
    }
  __syncthreads();   // zs and xa are free
}

// one colour sweep: cluster c of the launch owns SAP block blocks[c]
template <int RB, int RPL>
__global__ void __launch_bounds__(32 * SAPH_W, 2) k_csap_half(cplx<float>* __restrict__ z,
                                                                 const cplx<float>* __restrict__ bsrc,
                                                                 const __half2* __restrict__ blk,
                                                                 const float* __restrict__ bscale, Geom g, int n,
                                                                 FDiv fn, size_t rstride, int nrhs,
                                                                 const int* __restrict__ blocks, int k_mr, int spc,
                                                                 int nst, int* err, const int* __restrict__ bsite,
                                                                 const int* __restrict__ bloc) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  // the next sweep (launched with programmatic stream serialization) may stage its blocks while
  // this one runs; it waits for this grid before reading z or b
  pdl_launch_dependents();
  cg::cluster_group cluster = cg::this_cluster();
  const int CLS = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const SapHSmem L = saph_smem_layout(g.vB, n, spc, RB, nst * spc, 1);
  const __half2* stage = reinterpret_cast<const __half2*>(smem_raw);   // [spc][nst slots][n][n]
  const int* kof = reinterpret_cast<const int*>(smem_raw + L.kof);
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(smem_raw + L.bar);
  const int* own = bsite + (size_t)blocks[blockIdx.x / CLS] * g.vB + rank * spc;
  const int nn = n * n;
  if (threadIdx.x < 3) mbar_init(bar + threadIdx.x, 1);
  saph_tables(g, n, RB, own, spc, bloc, bscale, smem_raw, L, 0);
  cluster.sync();   // every CTA's exchange barriers are set up
  if (threadIdx.x < 32) {
    if (threadIdx.x == 0) mbar_arrive_expect_tx(bar, (unsigned)(spc * nst * nn * sizeof(__half2)));
    __syncwarp();
    for (int e = threadIdx.x; e < spc * nst; e += 32) {
      const int sl = e / nst;
      bulk_g2s(smem_raw + (size_t)e * nn * sizeof(__half2), blk + ((size_t)own[sl] * 9 + kof[sl * 9 + e - sl * nst]) * nn,
               (unsigned)(nn * sizeof(__half2)), bar);
    }
  }
  if (threadIdx.x == blockDim.x - 1) saph_links(n, RB, spc, rank, smem_raw, L, 0);
  pdl_wait();   // the previous kernel's z and b are complete from here on
  int ok = 1;
  unsigned seq = 0;
  for (int rh0 = 0; rh0 < nrhs; rh0 += RB)
    saph_block<RB, RPL, false>(
        cluster, z, bsrc, g.vB, n, fn, rstride, rh0, min(RB, nrhs - rh0), k_mr, spc, own, smem_raw, L, 0, seq, err,
        stage, nst, [&](int sl, int slot) { return blk + ((size_t)own[sl] * 9 + kof[sl * 9 + slot]) * nn; },
        [&] {
          if (rh0 == 0) {
            ok = __syncthreads_and(mbar_wait_bounded(bar, 0) ? 1 : 0);
            if (!ok && threadIdx.x == 0) atomicExch(err, 2);
          } else {
            __syncthreads();
          }
          return ok != 0;
        });
  if (!ok && threadIdx.x == 0) mbar_wait_bounded(bar, 0);   // no copy may still be in flight at exit
  cluster.sync();   // no CTA leaves while its last copies to others may still be read
}

// ---------------------------------------------------------------------------
// Persistent coarse SAP: all `iters` SAP applications (a red then a black sweep each) of one
// smoother call in one launch, for levels whose SAP blocks of both colours are resident at once.
// Cluster c owns nbpc red and nbpc black blocks; each CTA stages the blocks inside those SAP blocks of its
// sites once, for the whole call, and reads the others (hops leaving the block, for rho only) from L2.  A
// block is done by saph_block (same arithmetic, same order as a launch per sweep); sweeps are separated
// by a barrier over all clusters, which the cooperative launch makes safe (all CTAs co-resident).  z is
// read through L2 (ld.global.cg): values written by other SMs in the previous sweep are never taken from
// a stale L1 line.

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Barrier over the clusters of a persistent launch.  Rank 0 of every cluster counts its cluster
// in (the counter is zeroed before the launch; round r is complete at ncl * (r + 1)) and waits
// for the others; the wait is bounded (about a second at the maximum clock), after which
// *err = 3 and every CTA of the cluster gets false.
__device__ bool persist_grid_sync(unsigned* cnt, unsigned target, cg::cluster_group& cluster, int* flag, int* err) {
  cluster.sync();   // the sweep's writes of every CTA of the cluster precede the arrival
  if (cluster.block_rank() == 0 && threadIdx.x == 0) {
    __threadfence();
    atomicAdd(cnt, 1u);
    const long long t0 = clock64();
    int ok = 1;
    while (ld_acquire_gpu(cnt) < target) {
      if (clock64() - t0 > 2000000000LL) {
        ok = 0;
        atomicExch(err, 3);
        break;
      }
      __nanosleep(64);
    }
    *flag = ok;
  }
  cluster.sync();
  return *cluster.map_shared_rank(flag, 0) != 0;
}

template <int RPL>
__global__ void __launch_bounds__(32 * SAPH_W, 1) k_csap_half_persist(
    cplx<float>* __restrict__ z, const cplx<float>* __restrict__ bsrc, const __half2* __restrict__ blk,
    const float* __restrict__ bscale, Geom g, int n, FDiv fn, size_t rstride, int nrhs,
    const int* __restrict__ blocks0, int nb0, const int* __restrict__ blocks1, int nb1, int k_mr, int spc, int nsl,
    int nbpc, int iters, int* err,
    const int* __restrict__ bsite, const int* __restrict__ bloc, unsigned* gcnt) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  cg::cluster_group cluster = cg::this_cluster();
  const int CLS = (int)cluster.num_blocks();
  const int rank = (int)cluster.block_rank();
  const int cid = blockIdx.x / CLS;
  const unsigned ncl = gridDim.x / CLS;
  const int vB = g.vB, nn = n * n;
  const SapHSmem L = saph_smem_layout(vB, n, spc, 1, 2 * nbpc * spc * nsl, 2 * nbpc);
  __half2* stage = reinterpret_cast<__half2*>(smem_raw);   // [2][nbpc][spc][nsl slots][n][n]
  const int* kof = reinterpret_cast<const int*>(smem_raw + L.kof);   // [2 nbpc][spc][9]
  int* flag = reinterpret_cast<int*>(smem_raw + L.flag);
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(smem_raw + L.bar);
  // the own sites of block j of colour c (null: the cluster has none)
  auto own_of = [&](int c, int j) -> const int* {
    const int q = cid * nbpc + j;
    if (q >= (c ? nb1 : nb0)) return nullptr;
    return bsite + (size_t)(c ? blocks1 : blocks0)[q] * vB + rank * spc;
  };
  for (int cj = 0; cj < 2 * nbpc; ++cj)
    if (const int* own = own_of(cj / nbpc, cj % nbpc)) saph_tables(g, n, 1, own, spc, bloc, bscale, smem_raw, L, cj);
  if (threadIdx.x < 3) mbar_init(bar + threadIdx.x, 1);
  cluster.sync();   // every CTA's exchange barriers are set up
  if (threadIdx.x == blockDim.x - 1)
    for (int cj = 0; cj < 2 * nbpc; ++cj)
      if (own_of(cj / nbpc, cj % nbpc)) saph_links(n, 1, spc, rank, smem_raw, L, cj);
  if (threadIdx.x == 0) {   // nsl slots of every site: those inside the SAP block, then others up to that number
    int cnt = 0;
    for (int cj = 0; cj < 2 * nbpc; ++cj) cnt += own_of(cj / nbpc, cj % nbpc) ? spc * nsl : 0;
    mbar_arrive_expect_tx(bar, (unsigned)(cnt * nn * sizeof(__half2)));
    for (int cj = 0; cj < 2 * nbpc; ++cj)
      if (const int* own = own_of(cj / nbpc, cj % nbpc))
        for (int sl = 0; sl < spc; ++sl)
          for (int e = 0; e < nsl; ++e)
            bulk_g2s(stage + ((size_t)(cj * spc + sl) * nsl + e) * nn,
                     blk + ((size_t)own[sl] * 9 + kof[(cj * spc + sl) * 9 + e]) * nn, (unsigned)(nn * sizeof(__half2)),
                     bar);
  }
  const int ok = __syncthreads_and(mbar_wait_bounded(bar, 0) ? 1 : 0);
  if (!ok && threadIdx.x == 0) atomicExch(err, 2);
  unsigned round = 0, seq = 0;
  bool alive = true;
  for (int it = 0; it < iters && alive; ++it)
    for (int c = 0; c < 2 && alive; ++c) {
      for (int j = 0; j < nbpc; ++j) {
        const int cj = c * nbpc + j;
        const int* own = own_of(c, j);
        if (!own) continue;   // uniform over the cluster
        for (int rh = 0; rh < nrhs; ++rh)
          saph_block<1, RPL, true>(
              cluster, z, bsrc, vB, n, fn, rstride, rh, 1, k_mr, spc, own, smem_raw, L, cj, seq, err,
              (const __half2*)stage + (size_t)cj * spc * nsl * nn, nsl,
              [&](int sl, int slot) { return blk + ((size_t)own[sl] * 9 + kof[(cj * spc + sl) * 9 + slot]) * nn; },
              [&] {
                __syncthreads();
                return ok != 0;
              });
      }
      if (it + 1 < iters || c == 0) {
        ++round;
        alive = persist_grid_sync(gcnt, ncl * round, cluster, flag, err);
      }
    }
  if (!ok && threadIdx.x == 0) mbar_wait_bounded(bar, 0);   // no copy may still be in flight at exit
  cluster.sync();   // no CTA exits while others may still write into its shared memory
}

// Gauss-Jordan inversion with partial pivoting of every self block (FP64).
__global__ void k_selfinv_build(cplx<double>* __restrict__ inv, const cplx<double>* __restrict__ blk, int n,
                                int* err) {
  extern __shared__ unsigned char smem_raw[];
  cplx<double>* a = reinterpret_cast<cplx<double>*>(smem_raw);   // [n][2n] row-major
  cplx<double>* fac = a + (size_t)n * 2 * n;                       // [n] column k before elimination
  __shared__ int piv;
  const int site = blockIdx.x;
  const int w = 2 * n;
  for (int e = threadIdx.x; e < n * w; e += blockDim.x) {
    const int i = e / w, j = e % w;
    a[e] = j < n ? blk[bidx(site, 0, n, i, j)] : cmk(i == j - n ? 1.0 : 0.0, 0.0);
  }
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    if (threadIdx.x == 0) {
      int p = k;
      double best = cnorm2(a[k * w + k]);
      for (int i = k + 1; i < n; ++i) {
        const double v = cnorm2(a[i * w + k]);
        if (v > best) { best = v; p = i; }
      }
      piv = best > 0.0 ? p : -1;
    }
    __syncthreads();
    if (piv < 0) {
      if (threadIdx.x == 0) atomicExch(err, 1);
      return;
    }
    if (piv != k)
      for (int j = threadIdx.x; j < w; j += blockDim.x) {
        const cplx<double> t = a[k * w + j];
        a[k * w + j] = a[piv * w + j];
        a[piv * w + j] = t;
      }
    __syncthreads();
    const cplx<double> d = a[k * w + k];
    const double dn = cnorm2(d);
    const cplx<double> dinv = cmk(d.re / dn, -d.im / dn);
    __syncthreads();
    for (int j = threadIdx.x; j < w; j += blockDim.x) a[k * w + j] = a[k * w + j] * dinv;
    for (int i = threadIdx.x; i < n; i += blockDim.x) fac[i] = a[i * w + k];
    __syncthreads();
    for (int e = threadIdx.x; e < n * w; e += blockDim.x) {
      const int i = e / w, j = e % w;
      if (i != k) a[e] = a[e] - fac[i] * a[k * w + j];
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const int i = e % n, j = e / n;
    inv[((size_t)site * n + j) * n + i] = a[i * w + n + j];
  }
}

template <typename T>
__global__ void k_selfinv_apply(cplx<T>* __restrict__ out, const cplx<T>* __restrict__ in,
                                const cplx<T>* __restrict__ inv, Geom g, int n, int parity, size_t rstride) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (size_t)g.V * n) return;
  const int site = (int)(t / n), i = (int)(t % n);
  const size_t ro = (size_t)blockIdx.y * rstride;
  int c[4];
  geom_coords(g, site, c);
  cplx<T> acc = czero<T>();
  if (parity < 0 || geom_parity(c) == parity) {
    const cplx<T>* v = in + ro + (size_t)site * n;
    for (int j = 0; j < n; ++j) cfma(acc, inv[((size_t)site * n + j) * n + i], v[j]);
  }
  out[ro + t] = acc;
}

template <typename T>
__global__ void k_sub_parity(cplx<T>* y, const cplx<T>* a, const cplx<T>* b,
                             Geom g, int n, int parity, size_t rstride) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (size_t)g.V * n) return;
  const int site = (int)(t / n);
  const size_t ro = (size_t)blockIdx.y * rstride;
  int c[4];
  geom_coords(g, site, c);
  const bool keep = parity < 0 || geom_parity(c) == parity;
  y[ro + t] = keep ? a[ro + t] - (b ? b[ro + t] : czero<T>()) : czero<T>();
}

template <typename T>
__global__ void k_coarse_import(cplx<T>* __restrict__ dst, const cplx<double>* __restrict__ src, Geom g, int n,
                                size_t rstride) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (size_t)g.V * n) return;
  const int site = (int)(t / n), i = (int)(t % n);
  int c[4];
  geom_coords(g, site, c);
  const size_t lex = (size_t)lin4(c, g.L);
  dst[(size_t)blockIdx.y * rstride + t] = ccast<T>(src[(size_t)blockIdx.y * g.V * n + lex * n + i]);
}

template <typename T>
__global__ void k_coarse_export(cplx<double>* __restrict__ dst, const cplx<T>* __restrict__ src, Geom g, int n,
                                size_t rstride) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (size_t)g.V * n) return;
  const int site = (int)(t / n), i = (int)(t % n);
  int c[4];
  geom_coords(g, site, c);
  const size_t lex = (size_t)lin4(c, g.L);
  dst[(size_t)blockIdx.y * g.V * n + lex * n + i] = ccast<double>(src[(size_t)blockIdx.y * rstride + t]);
}

// internal [V][9][n][n] column-major  ->  ABI [lex][9][n][n] row-major
__global__ void k_blocks_export(cplx<double>* __restrict__ dst, const cplx<double>* __restrict__ blk, Geom g, int n) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t per = (size_t)9 * n * n;
  if (t >= (size_t)g.V * per) return;
  const int site = (int)(t / per);
  const size_t r = t % per;
  const int k = (int)(r / ((size_t)n * n));
  const int e = (int)(r % ((size_t)n * n));
  const int i = e / n, j = e % n;
  int c[4];
  geom_coords(g, site, c);
  const size_t lex = (size_t)lin4(c, g.L);
  dst[lex * per + (size_t)k * n * n + (size_t)i * n + j] = blk[bidx(site, k, n, i, j)];
}

// FP16 copy of one site's 9 blocks: s = float(max |re|, |im|), q = RNE_half(x / s) with x / s as the product
// with the reciprocal (as in the copy of P: FP64 divisions and comparisons would bound the kernel)
__global__ void k_blocks_to_half(__half2* __restrict__ dst, float* __restrict__ scale,
                                 const cplx<double>* __restrict__ blk, int n) {
  __shared__ unsigned long long sh[32];
  __shared__ double rs;
  const int per = 9 * n * n;
  const cplx<double>* src = blk + (size_t)blockIdx.x * per;
  unsigned long long mx = 0ull;
  for (int e = threadIdx.x; e < per; e += blockDim.x) mx = max(mx, max(abs_bits(src[e].re), abs_bits(src[e].im)));
  for (int off = 16; off >= 1; off >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, off));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) mx = max(mx, sh[w]);
    const double m = __longlong_as_double((long long)mx);
    const float sf = m > 0.0 ? (float)m : 1.0f;
    scale[blockIdx.x] = sf;
    rs = 1.0 / (double)sf;
  }
  __syncthreads();
  const double r = rs;
  __half2* d = dst + (size_t)blockIdx.x * per;
  for (int e = threadIdx.x; e < per; e += blockDim.x)
    d[e] = __halves2half2(__double2half(src[e].re * r), __double2half(src[e].im * r));
}

}  // namespace

namespace dd {

void blocks_to_half(__half2* dst, float* scale, const cplx<double>* blk, int V, int n, cudaStream_t st) {
  count_launch();
  k_blocks_to_half<<<V, 256, 0, st>>>(dst, scale, blk, n);
}

template <typename T>
void coarse_apply(cplx<T>* out, const cplx<T>* in, const cplx<T>* b, const CoarseOp<T>& op, int nrhs, size_t rstride,
                  int sel, int sel_mu, int in_chir, cudaStream_t st) {
  const int threads = ((9 * op.n + 31) / 32) * 32;
  const size_t sm = (size_t)18 * op.n * sizeof(cplx<T>);
  dim3 grid(op.g.V, nrhs);
  if constexpr (sizeof(T) == 4) {
    // the whole operator on FP16 storage: the tensor-core kernel where the autotuner chose it
    if (op.blkh && op.tc_ks > 0 && sel == SEL_FULL && in_chir < 0) {
      if (coarse_apply_tc(out, in, b, op, nrhs, rstride, op.tc_ks, st) == cudaSuccess) return;
      cudaGetLastError();
    }
  }
  count_launch();
  if constexpr (sizeof(T) == 4) {
    if (op.blkh) {
      if (b)
        k_coarse_apply<float, true, __half2><<<grid, threads, sm, st>>>(out, in, b, op.blkh, op.bscale, op.g, op.n,
                                                                         rstride, sel, sel_mu, in_chir);
      else
        k_coarse_apply<float, false, __half2><<<grid, threads, sm, st>>>(out, in, b, op.blkh, op.bscale, op.g, op.n,
                                                                          rstride, sel, sel_mu, in_chir);
      return;
    }
  }
  if (b)
    k_coarse_apply<T, true, cplx<T>><<<grid, threads, sm, st>>>(out, in, b, op.blk, nullptr, op.g, op.n, rstride, sel,
                                                                 sel_mu, in_chir);
  else
    k_coarse_apply<T, false, cplx<T>><<<grid, threads, sm, st>>>(out, in, b, op.blk, nullptr, op.g, op.n, rstride,
                                                                  sel, sel_mu, in_chir);
}

// staged blocks per site of the cluster SAP: the self block plus the hops that stay inside
// the SAP block, maximised over the sites of a block (every block has the same shape)
int coarse_sap_slots(const Geom& g) {
  int best = 1;
  for (int loc = 0; loc < g.vB; ++loc) {
    int c[4];
    delin4(loc, g.B, c);   // the sites of the block at the origin
    int cnt = 1;
    for (int k = 1; k < 9; ++k) cnt += hop_internal(g, c, (k - 1) % 4, k <= 4 ? +1 : -1, g.fB) ? 1 : 0;
    best = cnt > best ? cnt : best;
  }
  return best;
}

// The dynamic shared-memory limit of a kernel is a process-wide attribute: it is raised to the
// device maximum (not to this plan's size), so that a hierarchy set up later with smaller blocks
// cannot lower it below what an earlier hierarchy's launches use.
template <typename T>
void sap_cluster_attrs(size_t smem, int CLS) {
  if (cudaFuncSetAttribute(k_coarse_sap_cluster<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) !=
      cudaSuccess) {
    cudaGetLastError();
    cudaFuncSetAttribute(k_coarse_sap_cluster<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  }
  if (CLS > 8) cudaFuncSetAttribute(k_coarse_sap_cluster<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

// cluster plan of the coarse SAP on blocks in the compute precision: cluster size CLS, sites per CTA
// and staged blocks per site (0, and nothing written, if no plan fits).
template <typename T>
int coarse_sap_cluster_plan(const Geom& g, int n, int* CLS_out, int* spc_out, int* nsl_out, int prefer) {
  const int nsl = coarse_sap_slots(g);
  for (int CLS : {prefer, 16, 8, 4, 2}) {
    if (CLS != 2 && CLS != 4 && CLS != 8 && CLS != 16) continue;
    if (g.vB % CLS) continue;
    const int spc = g.vB / CLS;
    const int threads = ((9 * spc * n + 31) / 32) * 32;
    if (threads > 768) continue;   // launch bounds of k_coarse_sap_cluster
    const size_t sm = sap_smem_layout(g.vB, n, spc, nsl, sizeof(T)).total;
    if (sm > 227 * 1024) continue;
    sap_cluster_attrs<T>(sm, CLS);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CLS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(CLS, 1, 1);
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = sm;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int nclusters = 0;
    if (cudaOccupancyMaxActiveClusters(&nclusters, k_coarse_sap_cluster<T>, &cfg) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    if (nclusters < 1) continue;
    *CLS_out = CLS;
    *spc_out = spc;
    *nsl_out = nsl;
    return 1;
  }
  return 0;
}

// Persistent SAP on FP16 blocks (FP32 compute): the launch's shared memory and threads for nbpc
// SAP blocks of each colour per cluster, and whether all clusters (max(nb0, nb1) / nbpc of
// op.saph_cls CTAs) can be resident at once on this device.  Cluster size and staged blocks per site
// are those of the plan of the kernel on FP16 blocks (the other cluster kernel's plan refuses levels that
// this one takes); 0 without a plan that stages every block inside the SAP block, which the MR steps read.
size_t coarse_sap_persist_smem(const CoarseOp<float>& op, int nbpc) {
  if (op.saph_cls <= 0 || op.saph_nst < coarse_sap_slots(op.g)) return 0;
  const int spc = op.g.vB / op.saph_cls;
  return saph_smem_layout(op.g.vB, op.n, spc, 1, 2 * nbpc * spc * op.saph_nst, 2 * nbpc).total;
}

namespace {
int saph_threads(int rows, int n) { return 32 * saph_warps(rows, saph_rpl(n)); }
int saph_threads(const CoarseOp<float>& op) { return saph_threads(op.g.vB / op.saph_cls * op.n, op.n); }
template <int RB>
auto saph_kernel(int n) {
  const int r = saph_rpl(n);
  return r == 8 ? k_csap_half<RB, 8> : r == 4 ? k_csap_half<RB, 4> : k_csap_half<RB, 2>;
}
auto saph_persist_kernel(const CoarseOp<float>& op) {
  const int r = saph_rpl(op.n);
  return r == 8 ? k_csap_half_persist<8> : r == 4 ? k_csap_half_persist<4> : k_csap_half_persist<2>;
}
void saph_attrs(const void* fn) {   // process-wide limits: the device maximum
  cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  cudaGetLastError();
}
}  // namespace

// Cluster size and staged blocks per site (those inside the SAP block) of the kernel on FP16 blocks; 0 if none fits.
// Sixteen CTAs per SAP block where all blocks of a colour are then resident at once, else eight: 16 blocks per colour
// (16^3x32, 40 dof) 25.5 us per sweep with sixteen and 26.8 with eight, 34.0 and 37.4 for two right-hand sides;
// 128 blocks (32^4) 112 and 115, 377 and 271 for four right-hand sides.  Staging all nine blocks of a site: 25.0
// and 42, 148 and 204 for one right-hand side (fewer clusters fit).
int coarse_saph_plan(const Geom& g, int n, int nblocks, int* CLS_out, int* nst_out, int prefer) {
  *CLS_out = *nst_out = 0;
  const int nst = coarse_sap_slots(g);
  for (int pass = 0; pass < 2; ++pass)   // the second without the residency condition
    for (int CLS : {prefer, 16, 8, 4, 2}) {
      if ((CLS != 2 && CLS != 4 && CLS != 8 && CLS != 16) || g.vB % CLS) continue;
      const int spc = g.vB / CLS, rows = spc * n;
      const size_t sm = saph_smem_layout(g.vB, n, spc, 1, nst * spc, 1).total;
      if (sm > 227 * 1024 || spc > SAPH_SITES) continue;
      const void* fn = (const void*)saph_kernel<1>(n);
      saph_attrs(fn);
      saph_attrs((const void*)saph_kernel<2>(n));
      cudaLaunchConfig_t cfg = {};
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = CLS;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg.gridDim = dim3(CLS, 1, 1);
      cfg.blockDim = dim3(saph_threads(rows, n), 1, 1);
      cfg.dynamicSmemBytes = sm;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      int nclusters = 0;
      if (cudaOccupancyMaxActiveClusters(&nclusters, fn, &cfg) != cudaSuccess || nclusters < 1) {
        cudaGetLastError();
        continue;
      }
      if (pass == 0 && CLS == 16 && CLS != prefer && nclusters < nblocks) continue;
      *CLS_out = CLS;
      *nst_out = nst;
      return 1;
    }
  return 0;
}

bool coarse_sap_persist_fits(const CoarseOp<float>& op, int nb0, int nb1, int* max_clusters, int* nbpc_out,
                             int min_nbpc) {
  if (max_clusters) *max_clusters = -1;
  if (nbpc_out) *nbpc_out = 0;
  if (op.saph_cls <= 0 || !op.blkh || nb0 <= 0 || nb1 <= 0) return false;
  const int CLS = op.saph_cls;
  const int nb = nb0 > nb1 ? nb0 : nb1;
  for (int nbpc = min_nbpc < 1 ? 1 : min_nbpc; nbpc <= 2; ++nbpc) {
    const int threads = saph_threads(op);
    const size_t sm = coarse_sap_persist_smem(op, nbpc);
    if (sm == 0 || sm > 227 * 1024) continue;
    const void* fn = (const void*)saph_persist_kernel(op);
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             227 * 1024) != cudaSuccess ||   // process-wide limit: the device maximum
        (CLS > 8 && cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)) {
      cudaGetLastError();
      continue;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CLS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(CLS, 1, 1);
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = sm;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int nclusters = 0;
    if (cudaOccupancyMaxActiveClusters(&nclusters, fn, &cfg) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    if (max_clusters) *max_clusters = nclusters;
    if (nclusters >= (nb + nbpc - 1) / nbpc) {
      if (nbpc_out) *nbpc_out = nbpc;
      return true;
    }
  }
  return false;
}

cudaError_t coarse_sap_persist(cplx<float>* z, const cplx<float>* b, const CoarseOp<float>& op, const int* blocks0,
                               int nb0, const int* blocks1, int nb1, int nrhs, size_t rstride, int k_mr, int iters,
                               int nbpc, unsigned* gcnt, cudaStream_t st) {
  if (nrhs <= 0 || iters <= 0) return cudaSuccess;
  if (!op.blkh || nb0 <= 0 || nb1 <= 0 || nbpc < 1 || nbpc > 2) return cudaErrorInvalidValue;
  const size_t sm = coarse_sap_persist_smem(op, nbpc);
  if (sm == 0) return cudaErrorInvalidValue;
  const int CLS = op.saph_cls, spc = op.g.vB / CLS;
  const int nb = nb0 > nb1 ? nb0 : nb1;
  cudaError_t e = cudaMemsetAsync(gcnt, 0, sizeof(unsigned), st);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CLS;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeCooperative;   // all clusters co-resident (they wait on one another)
  attr[1].val.cooperative = 1;
  cfg.gridDim = dim3(((nb + nbpc - 1) / nbpc) * CLS, 1, 1);
  cfg.blockDim = dim3(saph_threads(op), 1, 1);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  count_launch();
  return cudaLaunchKernelEx(&cfg, saph_persist_kernel(op), z, b, op.blkh, op.bscale, op.g, op.n, fdiv_make(op.n), rstride, nrhs, blocks0, nb0,
                            blocks1, nb1, k_mr, spc, op.saph_nst, nbpc, iters, op.err, op.bsite,
                            op.bloc, gcnt);
}

template <typename T>
cudaError_t coarse_sap_sweep(cplx<T>* z, const cplx<T>* b, const CoarseOp<T>& op, const int* blocks, int nblocks,
                             int nrhs, size_t rstride, int k_mr, cudaStream_t st) {
  const int cls = sizeof(T) == 4 && op.blkh ? op.saph_cls : op.sap_cls;
  if (cls > 0) {
    const int spc = op.g.vB / cls;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cls;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    // consecutive colour sweeps: the next one stages its blocks while this one finishes
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(nblocks * cls, 1, 1);   // one cluster per SAP block loops over the batch
    cfg.stream = st;
    cfg.attrs = attr;
    count_launch();
    // with programmatic serialization first, then (if the attribute is refused) without it
    for (int na = 2; na >= 1; --na) {
      cfg.numAttrs = na;
      cudaError_t e;
      if constexpr (sizeof(T) == 4) {
        if (op.blkh) {
          // two right-hand sides at a time unless that costs the second CTA per SM (a right-hand side's
          // arithmetic does not depend on it)
          auto smem = [&](int rb) { return saph_smem_layout(op.g.vB, op.n, spc, rb, op.saph_nst * spc, 1).total; };
          const size_t two_per_sm = 113 * 1024;
          const int rb = nrhs > 1 && smem(2) <= 227 * 1024 && (smem(2) <= two_per_sm || smem(1) > two_per_sm) ? 2 : 1;
          cfg.blockDim = dim3(saph_threads(op), 1, 1);
          cfg.dynamicSmemBytes = smem(rb);
          e = cudaLaunchKernelEx(&cfg, rb == 2 ? saph_kernel<2>(op.n) : saph_kernel<1>(op.n), z, b,
                                 op.blkh, op.bscale, op.g, op.n, fdiv_make(op.n), rstride, nrhs, blocks, k_mr, spc, op.saph_nst, op.err,
                                 op.bsite, op.bloc);
          if (e == cudaSuccess) return cudaSuccess;
          cudaGetLastError();
          continue;
        }
      }
      cfg.blockDim = dim3(((9 * spc * op.n + 31) / 32) * 32, 1, 1);
      cfg.dynamicSmemBytes = sap_smem_layout(op.g.vB, op.n, spc, op.sap_nsl, sizeof(T)).total;
      e = cudaLaunchKernelEx(&cfg, k_coarse_sap_cluster<T>, z, b, (const cplx<T>*)op.blk, op.g, op.n, rstride, nrhs,
                             blocks, k_mr, spc, op.sap_nsl, op.err, op.bsite, op.bloc);
      if (e == cudaSuccess) return cudaSuccess;
      cudaGetLastError();
    }
    // cluster launch refused: run the one-CTA-per-block kernel instead
  }
  // one CTA per SAP block with rpt rows per thread: the fewest of 1, 4, 8 for which
  // the CTA stays within the threads the kernel's registers allow
  const int rows = op.g.vB * op.n;
  const size_t sm = (size_t)rows * sizeof(cplx<T>) + 32 * 3 * sizeof(T);
  const bool half = sizeof(T) == 4 && op.blkh;
  // threads per CTA the kernel's registers allow, queried once per variant (a property of the
  // compiled kernel, the same on every device of this architecture); the entries are atomics
  // because serving workers launch from several host threads
  static std::atomic<int> maxthr[2][2][3];   // [FP64][FP16 blocks][rpt 1, 4, 8]; 0 = not queried
  static DeviceOnce once[2][2][3];
  std::atomic<int>* mt = maxthr[sizeof(T) == 8][half ? 1 : 0];
  auto query = [&](const void* fn, int q) {
    raise_smem_limit(once[sizeof(T) == 8][half ? 1 : 0][q], fn);
    int v = mt[q].load(std::memory_order_acquire);
    if (v == 0) {
      cudaFuncAttributes a;
      v = cudaFuncGetAttributes(&a, fn) == cudaSuccess ? a.maxThreadsPerBlock : -1;
      cudaGetLastError();
      mt[q].store(v, std::memory_order_release);
    }
    return v;
  };
  const void* fns[3];
  if constexpr (sizeof(T) == 4) {
    if (half) {
      fns[0] = (const void*)k_coarse_sap<float, __half2, 1>;
      fns[1] = (const void*)k_coarse_sap<float, __half2, 4>;
      fns[2] = (const void*)k_coarse_sap<float, __half2, 8>;
    }
  }
  if (!half) {
    fns[0] = (const void*)k_coarse_sap<T, cplx<T>, 1>;
    fns[1] = (const void*)k_coarse_sap<T, cplx<T>, 4>;
    fns[2] = (const void*)k_coarse_sap<T, cplx<T>, 8>;
  }
  const int rpts[3] = {1, 4, 8};
  int q = 2;
  for (int c = 0; c < 3; ++c)
    if (((div_up(rows, rpts[c]) + 31) / 32) * 32 <= query(fns[c], c)) {
      q = c;
      break;
    }
  const int threads = ((div_up(rows, rpts[q]) + 31) / 32) * 32;
  if (threads > query(fns[q], q)) return cudaErrorInvalidConfiguration;   // block too large even at 8 rows
  count_launch();
  const dim3 grid(nblocks, nrhs);
  if constexpr (sizeof(T) == 4) {
    if (half) {
      if (q == 0)
        k_coarse_sap<float, __half2, 1><<<grid, threads, sm, st>>>(z, b, op.blkh, op.bscale, op.g, op.n, rstride,
                                                                    blocks, k_mr, op.bsite, op.bloc);
      else if (q == 1)
        k_coarse_sap<float, __half2, 4><<<grid, threads, sm, st>>>(z, b, op.blkh, op.bscale, op.g, op.n, rstride,
                                                                    blocks, k_mr, op.bsite, op.bloc);
      else
        k_coarse_sap<float, __half2, 8><<<grid, threads, sm, st>>>(z, b, op.blkh, op.bscale, op.g, op.n, rstride,
                                                                    blocks, k_mr, op.bsite, op.bloc);
      return cudaPeekAtLastError();
    }
  }
  if (q == 0)
    k_coarse_sap<T, cplx<T>, 1><<<grid, threads, sm, st>>>(z, b, op.blk, nullptr, op.g, op.n, rstride, blocks, k_mr,
                                                            op.bsite, op.bloc);
  else if (q == 1)
    k_coarse_sap<T, cplx<T>, 4><<<grid, threads, sm, st>>>(z, b, op.blk, nullptr, op.g, op.n, rstride, blocks, k_mr,
                                                            op.bsite, op.bloc);
  else
    k_coarse_sap<T, cplx<T>, 8><<<grid, threads, sm, st>>>(z, b, op.blk, nullptr, op.g, op.n, rstride, blocks, k_mr,
                                                            op.bsite, op.bloc);
  return cudaPeekAtLastError();
}

template <typename T>
void coarse_schur_odd(cplx<T>* t, const cplx<T>* x, const cplx<T>* b, const CoarseOp<T>& op, double a, double c,
                      int nrhs, size_t rstride, cudaStream_t st) {
  const int threads = ((8 * op.n + 31) / 32) * 32;
  const size_t sm = (size_t)17 * op.n * sizeof(cplx<T>);
  count_launch();
  if constexpr (sizeof(T) == 4) {
    if (op.blkh) {
      k_schur_odd<float, __half2><<<dim3(op.n_odd, nrhs), threads, sm, st>>>(t, x, b, op.blkh, op.bscale, op.selfinv,
                                                                             op.odd_sites, op.g, op.n, rstride, a, c);
      return;
    }
  }
  k_schur_odd<T, cplx<T>><<<dim3(op.n_odd, nrhs), threads, sm, st>>>(t, x, b, op.blk, nullptr, op.selfinv,
                                                                      op.odd_sites, op.g, op.n, rstride, a, c);
}

template <typename T>
void coarse_schur_even(cplx<T>* y, const cplx<T>* x, const cplx<T>* t, const cplx<T>* b, const CoarseOp<T>& op,
                       double a, double s, double c, int nrhs, size_t rstride, cudaStream_t st) {
  const int threads = ((9 * op.n + 31) / 32) * 32;
  const size_t sm = (size_t)18 * op.n * sizeof(cplx<T>);
  count_launch();
  if constexpr (sizeof(T) == 4) {
    if (op.blkh) {
      k_schur_even<float, __half2><<<dim3(op.g.V, nrhs), threads, sm, st>>>(y, x, t, b, op.blkh, op.bscale, op.g, op.n,
                                                                            rstride, a, s, c);
      return;
    }
  }
  k_schur_even<T, cplx<T>><<<dim3(op.g.V, nrhs), threads, sm, st>>>(y, x, t, b, op.blk, nullptr, op.g, op.n, rstride,
                                                                     a, s, c);
}

void coarse_selfinv_build(cplx<double>* inv, const cplx<double>* blk, int V, int n, int* err, cudaStream_t st) {
  const size_t sm = ((size_t)n * 2 * n + n) * sizeof(cplx<double>);
  static DeviceOnce once;
  raise_smem_limit(once, (const void*)k_selfinv_build);
  count_launch();
  k_selfinv_build<<<V, 256, sm, st>>>(inv, blk, n, err);
}

template <typename T>
void coarse_selfinv_apply(cplx<T>* out, const cplx<T>* in, const CoarseOp<T>& op, int parity, int nrhs, size_t rstride,
                          cudaStream_t st) {
  const size_t tot = (size_t)op.g.V * op.n;
  count_launch();
  k_selfinv_apply<T><<<dim3(div_up(tot, 128), nrhs), 128, 0, st>>>(out, in, op.selfinv, op.g, op.n, parity, rstride);
}

template <typename T>
void coarse_sub_parity(cplx<T>* y, const cplx<T>* a, const cplx<T>* b, const Geom& g, int n, int parity, int nrhs,
                       size_t rstride, cudaStream_t st) {
  const size_t tot = (size_t)g.V * n;
  count_launch();
  k_sub_parity<T><<<dim3(div_up(tot, 128), nrhs), 128, 0, st>>>(y, a, b, g, n, parity, rstride);
}

template <typename T>
void coarse_import(cplx<T>* dst, const cplx<double>* src, const Geom& g, int n, int nrhs, size_t rstride,
                   cudaStream_t st) {
  count_launch();
  k_coarse_import<T><<<dim3(div_up((size_t)g.V * n, 128), nrhs), 128, 0, st>>>(dst, src, g, n, rstride);
}

template <typename T>
void coarse_export(cplx<double>* dst, const cplx<T>* src, const Geom& g, int n, int nrhs, size_t rstride,
                   cudaStream_t st) {
  count_launch();
  k_coarse_export<T><<<dim3(div_up((size_t)g.V * n, 128), nrhs), 128, 0, st>>>(dst, src, g, n, rstride);
}

void coarse_blocks_export(cplx<double>* dst, const cplx<double>* blk, const Geom& g, int n, cudaStream_t st) {
  count_launch();
  k_blocks_export<<<div_up((size_t)g.V * 9 * n * n, 128), 128, 0, st>>>(dst, blk, g, n);
}

#define INST(T)                                                                                                   \
  template void coarse_apply<T>(cplx<T>*, const cplx<T>*, const cplx<T>*, const CoarseOp<T>&, int, size_t, int,     \
                                int, int, cudaStream_t);                                                          \
  template void coarse_schur_odd<T>(cplx<T>*, const cplx<T>*, const cplx<T>*, const CoarseOp<T>&, double, double, \
                                    int, size_t, cudaStream_t);                                                   \
  template void coarse_schur_even<T>(cplx<T>*, const cplx<T>*, const cplx<T>*, const cplx<T>*, const CoarseOp<T>&, \
                                     double, double, double, int, size_t, cudaStream_t);                          \
  template int coarse_sap_cluster_plan<T>(const Geom&, int, int*, int*, int*, int);                                \
  template cudaError_t coarse_sap_sweep<T>(cplx<T>*, const cplx<T>*, const CoarseOp<T>&, const int*, int, int, size_t,   \
                                    int, cudaStream_t);                                                           \
  template void coarse_selfinv_apply<T>(cplx<T>*, const cplx<T>*, const CoarseOp<T>&, int, int, size_t,           \
                                        cudaStream_t);                                                            \
  template void coarse_sub_parity<T>(cplx<T>*, const cplx<T>*, const cplx<T>*, const Geom&, int, int, int, size_t, \
                                     cudaStream_t);                                                               \
  template void coarse_import<T>(cplx<T>*, const cplx<double>*, const Geom&, int, int, size_t, cudaStream_t);      \
  template void coarse_export<T>(cplx<double>*, const cplx<T>*, const Geom&, int, int, size_t, cudaStream_t);
INST(float)
INST(double)
#undef INST

}  // namespace dd
