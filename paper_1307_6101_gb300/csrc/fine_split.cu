// Fine-level FP64 kernels that share a site among six threads.
//
// GB300 executes about 3.5 FP64 FMAs per nanosecond and SM, and one warp alone gets a quarter of that
// (a DFMA of one warp issues every 31 ns, whether 16 or 32 of its lanes are active).  With one thread
// per site a small lattice therefore runs on a few SMs at their FP64 rate while the others idle, or on
// single warps at a quarter of it.  Here thread (site, s, a) owns colour a of the spins s and s + 2
// (s = 0, 1): for each hop it projects its component of the half spinor, the three colours of a
// half spinor meet in shared memory, and it multiplies its row of the link.  No product or sum is
// computed twice, so the operation count is that of one thread per site, on six times the threads.
//
// With gamma_mu = [[0, -Q], [-Q^+, 0]] a forward hop (1 - gamma_mu) projects h = up + Q dn and
// reconstructs low = Q^+ h, a backward hop has -Q; Q couples spin s to one lower spin with a
// phase q: t: -1, z: +i / -i (s = 0 / 1), lower spin s; y: +1 / -1, x: +i, lower spin 1 - s.
#include <cooperative_groups.h>

#include "common.cuh"
#include "kernels.h"

namespace cg = cooperative_groups;

namespace {

DD_HD int herm_pos(int i, int j) { return 6 + 2 * (i * 6 - (i * (i + 1)) / 2 + (j - i - 1)); }

// sign of the phase of Q for (mu, s): real for mu = t, y, imaginary for z, x
__device__ __forceinline__ double phase_sign(int mu, int s) {
  return mu == 0 ? -1.0 : (mu == 3 || s == 0) ? 1.0 : -1.0;
}

// component (s, a) of the projected half spinor of a hop: up + q dn, negated if neg
__device__ __forceinline__ cplx<double> project(int mu, double q, cplx<double> up, cplx<double> dn, bool neg) {
  cplx<double> h;
  if (mu == 0 || mu == 2) h = cmk(fma(q, dn.re, up.re), fma(q, dn.im, up.im));
  else h = cmk(fma(-q, dn.im, up.re), fma(q, dn.re, up.im));
  return neg ? cmk(-h.re, -h.im) : h;
}

// acc += conj(q) g for the phase of (mu, s)
__device__ __forceinline__ void reconstruct(int mu, double q, cplx<double> g, cplx<double>& acc) {
  if (mu == 0 || mu == 2) acc = cmk(fma(q, g.re, acc.re), fma(q, g.im, acc.im));
  else acc = cmk(fma(q, g.im, acc.re), fma(-q, g.re, acc.im));
}

// row a of U_mu(x) (forward) or of U_mu(n)^+ (backward) times the half spinor h[0], h[hs], h[2 hs]
__device__ __forceinline__ cplx<double> link_row(const cplx<double>* __restrict__ U, int V, int mu, bool fwd, int site,
                                                 int a, const cplx<double>* h, int hs) {
  const cplx<double>* u = U + (size_t)(mu * 9 + (fwd ? 3 * a : a)) * V + site;
  const size_t st = (size_t)(fwd ? 1 : 3) * V;
  cplx<double> g = czero<double>();
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    cplx<double> e = u[b * st];
    if (!fwd) e.im = -e.im;
    cfma(g, e, h[b * hs]);
  }
  return g;
}

// row i of the packed Hermitian block of one chirality (clov at the site, stride V) times v[0], v[vs], ...
__device__ __forceinline__ cplx<double> clover_row(const double* __restrict__ clov, size_t V, int i,
                                                   const cplx<double>* v, size_t vs) {
  const cplx<double> vi = v[i * vs];
  const double d = clov[i * V];
  cplx<double> w = cmk(d * vi.re, d * vi.im);
#pragma unroll
  for (int k = 1; k < 6; ++k) {
    const int j = i + k < 6 ? i + k : i + k - 6;   // the five other columns
    const int p = i < j ? herm_pos(i, j) : herm_pos(j, i);
    const double im = clov[(size_t)(p + 1) * V];
    cfma(w, cmk(clov[(size_t)p * V], i < j ? im : -im), v[j * vs]);
  }
  return w;
}

// sums of three values over the warp: lanes 0, 8 and 16 return them.  The lanes share the values out as
// they fold (six additions; one butterfly per value takes fifteen)
__device__ __forceinline__ double warp_sum3(const double v[3], int lane) {
  const bool h16 = (lane & 16) != 0, h8 = (lane & 8) != 0;
  double a = (h16 ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, h16 ? v[0] : v[2], 16);
  double b = (h16 ? 0.0 : v[1]) + __shfl_xor_sync(0xffffffffu, h16 ? v[1] : 0.0, 16);
  a = (h8 ? b : a) + __shfl_xor_sync(0xffffffffu, h8 ? a : b, 8);
#pragma unroll
  for (int off = 4; off >= 1; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
  return a;
}

struct Hop {
  int n;        // neighbour (global site index, or position in the SAP block)
  bool on, fwd;
};

// out = D in (or b - D in): 32 sites per CTA of 192 threads.  Shared memory: the projected components
// [8 hops][6][32] and the lower-spin sums of the partner spin [6][32].  Bound by the FP64 rate (1152
// FP64 instructions per site) on every lattice that fills the chip, where it takes what one thread per
// site takes (ddamg_apply on 24^3x48 1634 us against 1646, 16^3x32 351 against 358), and faster below
// (16^4 198 against 219, 12^4 95 against 125, 8^4 51 against 84 of which 33 are the call's other work).
constexpr int DS = 32;

template <bool RESID>
__global__ void __launch_bounds__(6 * DS) k_fine_dslash_split(cplx<double>* __restrict__ out,
                                                              const cplx<double>* __restrict__ in,
                                                              const cplx<double>* __restrict__ bsrc,
                                                              const cplx<double>* __restrict__ U,
                                                              const double* __restrict__ clov, Geom g, int bc_t,
                                                              size_t rstride) {
  __shared__ cplx<double> H[8][6][DS];
  __shared__ cplx<double> X[6][DS];
  const int V = g.V;
  const int comp = threadIdx.x / DS, l = threadIdx.x % DS;
  const int s = comp / 3, a = comp % 3;
  const int x = blockIdx.x * DS + l;
  const bool active = x < V;
  const cplx<double>* pin = in + (size_t)blockIdx.y * rstride;
  int c[4] = {0, 0, 0, 0}, nb[8];
  if (active) geom_coords(g, x, c);
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int mu = k >> 1;
    nb[k] = active ? geom_neighbor(g, c, mu, (k & 1) ? -1 : +1) : 0;
    const double q = (k & 1) ? -phase_sign(mu, s) : phase_sign(mu, s);
    const bool neg = mu == 0 && bc_t < 0 && ((k & 1) ? c[0] == 0 : c[0] == g.L[0] - 1);
    const int ls = mu >= 2 ? 1 - s : s;
    H[k][comp][l] = project(mu, q, pin[(size_t)comp * V + nb[k]], pin[(size_t)(6 + 3 * ls + a) * V + nb[k]], neg);
  }
  __syncthreads();
  cplx<double> up = czero<double>(), lo = czero<double>(), lx = czero<double>();
  if (active) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int mu = k >> 1;
      const bool fwd = (k & 1) == 0;
      const double q = fwd ? phase_sign(mu, s) : -phase_sign(mu, s);
      const cplx<double> gr = link_row(U, V, mu, fwd, fwd ? x : nb[k], a, &H[k][3 * s][l], DS);
      up = up + gr;
      reconstruct(mu, q, gr, mu >= 2 ? lx : lo);
    }
  }
  X[comp][l] = lx;
  __syncthreads();
  if (!active) return;
  lo = lo + X[comp < 3 ? comp + 3 : comp - 3][l];
  const cplx<double> du = clover_row(clov + x, V, comp, pin + x, V);
  const cplx<double> dl = clover_row(clov + (size_t)36 * V + x, V, comp, pin + (size_t)6 * V + x, V);
  const size_t o = (size_t)blockIdx.y * rstride + (size_t)comp * V + x;
  cplx<double> ru = cmk(fma(-0.5, up.re, du.re), fma(-0.5, up.im, du.im));
  cplx<double> rl = cmk(fma(-0.5, lo.re, dl.re), fma(-0.5, lo.im, dl.im));
  if (RESID) {
    ru = bsrc[o] - ru;
    rl = bsrc[o + (size_t)6 * V] - rl;
  }
  out[o] = ru;
  out[o + (size_t)6 * V] = rl;
}

// One colour sweep of SAP (same method as k_fine_sap): one cluster of CLS CTAs per SAP block and
// right-hand side, CTA q owning S = ceil(vB / CLS) consecutive sites, six threads per site.  The block
// residual is spread over the CTAs' shared memory, and a hop into another CTA's sites reads it there.
// A site has at most two hops per direction inside its block.  They are done in two passes: the first
// takes the forward hop, or the backward one where only that is inside, the second the backward hop
// where both are; blocks of extent 2 need no second pass in that direction, so no warp runs a hop
// for half of its lanes.  Bound by the FP64 rate, and on small lattices by one warp's 31 ns per DFMA
// (three warps per SM at 2^4 blocks): 4 MR steps on 8^4 with 2^4 blocks 58 us per sweep (k_fine_sap, 8 CTAs:
// 516), 16^3x32 800 (1050).
constexpr int MAXCLS = 8;
constexpr int SMS = 152;   // of a GB300

template <int NT>   // most threads of a CTA
__global__ void __launch_bounds__(NT, 768 / NT) k_fine_sap_split(cplx<double>* __restrict__ z,
                                                        const cplx<double>* __restrict__ bsrc,
                                                        const cplx<double>* __restrict__ U,
                                                        const double* __restrict__ clov, Geom g, int bc_t,
                                                        size_t rstride, const int* __restrict__ blocks, int k_mr,
                                                        int S) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cg::cluster_group cluster = cg::this_cluster();
  const int CLS = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  cplx<double>* Rs = reinterpret_cast<cplx<double>*>(smem_raw);   // [12][S] residual of the own sites
  cplx<double>* H = Rs + 12 * S;                                   // [8][6][S] projected half spinors
  cplx<double>* X = H + 48 * S;                                    // [6][S] lower-spin sums of the partner
  double* red = reinterpret_cast<double*>(X + 6 * S);              // [24][3] warp partials
  double* cpart = red + 72;                                        // [2][MAXCLS][3] CTA partials
  short* nin = reinterpret_cast<short*>(cpart + 6 * MAXCLS);       // [8][S] hops inside the block
  const int V = g.V, vB = g.vB;
  const int blk = blocks[blockIdx.x / CLS];
  const int comp = threadIdx.x / S, l = threadIdx.x - comp * S;
  const int s = comp < 6 ? comp / 3 : 0, a = comp % 3;
  const int loc = rank * S + l;
  const bool active = comp < 6 && loc < vB;
  const int x = blk * vB + loc;
  const size_t ro = (size_t)blockIdx.y * rstride;
  cplx<double>* pz = z + ro;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  bool wrap_f, wrap_b;
  {
    int c[4] = {0, 0, 0, 0};
    if (active) geom_coords(g, x, c);
    wrap_f = bc_t < 0 && c[0] == g.L[0] - 1;
    wrap_b = bc_t < 0 && c[0] == 0;
    // per site and hop (mu, pass): 2 * position in the block of the neighbour + forward; -1: none
    if (active && comp == 0)
#pragma unroll 1
      for (int mu = 0; mu < 4; ++mu) {
        const bool f = hop_internal(g, c, mu, +1, g.fB), b = hop_internal(g, c, mu, -1, g.fB);
        nin[2 * mu * S + l] =
            f || b ? (short)(2 * (geom_neighbor(g, c, mu, f ? +1 : -1) - blk * vB) + (f ? 1 : 0)) : (short)-1;
        nin[(2 * mu + 1) * S + l] = f && b ? (short)(2 * (geom_neighbor(g, c, mu, -1) - blk * vB)) : (short)-1;
      }
  }
  // D v at the own components: hop(mu, pass) says which hops are on, get(component, n) reads v
  // at a neighbour, own(component) points at v's component at the own site (stride os)
  auto apply = [&](auto hop, auto get, const cplx<double>* own, size_t os, bool full, cplx<double>& pu,
                   cplx<double>& pl) {
    if (comp < 6) {
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int mu = k >> 1;
        const Hop hp = hop(mu, k & 1);
        if (hp.on) {
          const double q = hp.fwd ? phase_sign(mu, s) : -phase_sign(mu, s);
          const int ls = mu >= 2 ? 1 - s : s;
          H[(size_t)(k * 6 + comp) * S + l] =
              project(mu, q, get(comp, hp.n), get(6 + 3 * ls + a, hp.n), mu == 0 && (hp.fwd ? wrap_f : wrap_b));
        }
      }
    }
    __syncthreads();
    cplx<double> up = czero<double>(), lo = czero<double>(), lx = czero<double>();
    if (active) {
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int mu = k >> 1;
        // no site of a block has a second inside hop in a direction of extent 2 that does not wrap
        if (!full && (g.B[mu] == 1 || ((k & 1) && g.B[mu] == 2)) && g.B[mu] != g.L[mu]) continue;
        const Hop hp = hop(mu, k & 1);
        if (!hp.on) continue;
        const double q = hp.fwd ? phase_sign(mu, s) : -phase_sign(mu, s);
        const int site = hp.fwd ? x : (full ? hp.n : blk * vB + hp.n);
        const cplx<double> gr = link_row(U, V, mu, hp.fwd, site, a, H + (size_t)(k * 6 + 3 * s) * S + l, S);
        up = up + gr;
        reconstruct(mu, q, gr, mu >= 2 ? lx : lo);
      }
      X[(size_t)comp * S + l] = lx;
    }
    __syncthreads();
    if (active) {
      lo = lo + X[(size_t)(comp < 3 ? comp + 3 : comp - 3) * S + l];
      pu = clover_row(clov + x, V, comp, own, os);
      pl = clover_row(clov + (size_t)36 * V + x, V, comp, own + 6 * os, os);
      pu = cmk(fma(-0.5, up.re, pu.re), fma(-0.5, up.im, pu.im));
      pl = cmk(fma(-0.5, lo.re, pl.re), fma(-0.5, lo.im, pl.im));
    }
  };
  cplx<double> pu = czero<double>(), pl = czero<double>(), ru = czero<double>(), rl = czero<double>();
  cplx<double> xu = czero<double>(), xl = czero<double>();
  // rho = b - D z
  int c[4] = {0, 0, 0, 0};
  if (active) geom_coords(g, x, c);
  apply([&](int mu, int k) { return Hop{active ? geom_neighbor(g, c, mu, k ? -1 : +1) : 0, active, k == 0}; },
        [&](int f, int n) { return pz[(size_t)f * V + n]; }, pz + x, (size_t)V, true, pu, pl);
  if (active) {
    ru = bsrc[ro + (size_t)comp * V + x] - pu;
    rl = bsrc[ro + (size_t)(comp + 6) * V + x] - pl;
    Rs[(size_t)comp * S + l] = ru;
    Rs[(size_t)(comp + 6) * S + l] = rl;
  }
  if (CLS > 1) cluster.sync();
  else __syncthreads();
  auto inside = [&](int mu, int k) {
    const int n = active ? nin[(2 * mu + k) * S + l] : -1;
    return Hop{n >> 1, n >= 0, (n & 1) != 0};
  };
  auto get_r = [&](int f, int n) {
    if (CLS == 1) return Rs[(size_t)f * S + n];
    const int qr = n / S;
    return cluster.map_shared_rank(Rs, qr)[(size_t)f * S + (n - qr * S)];
  };
  for (int it = 0; it < k_mr; ++it) {
    apply(inside, get_r, Rs + l, (size_t)S, false, pu, pl);
    double v[3] = {0.0, 0.0, 0.0};
    if (active) {
      cdotc_acc(v[0], v[1], pu, ru);
      cdotc_acc(v[0], v[1], pl, rl);
      cnorm2_acc(v[2], pu);
      cnorm2_acc(v[2], pl);
    }
    const double vs = warp_sum3(v, lane);
    if (lane == 0 || lane == 8 || lane == 16) red[3 * warp + (lane >> 3)] = vs;
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 3; ++e) v[e] = 0.0;
    if (CLS == 1) {
      for (int w = 0; w < nw; ++w)
#pragma unroll
        for (int e = 0; e < 3; ++e) v[e] += red[3 * w + e];
    } else {
      double* cp = cpart + (it & 1) * 3 * MAXCLS;
      if (threadIdx.x < 3) {
        double t = 0.0;
        for (int w = 0; w < nw; ++w) t += red[3 * w + threadIdx.x];
        for (int q = 0; q < CLS; ++q) cluster.map_shared_rank(cp, q)[3 * rank + threadIdx.x] = t;
      }
      cluster.sync();
      for (int q = 0; q < CLS; ++q)
#pragma unroll
        for (int e = 0; e < 3; ++e) v[e] += cp[3 * q + e];
    }
    const cplx<double> alpha = v[2] > 0.0 ? cmk(v[0] / v[2], v[1] / v[2]) : czero<double>();
    cfma(xu, alpha, ru);
    cfma(xl, alpha, rl);
    ru = ru - alpha * pu;
    rl = rl - alpha * pl;
    if (active) {
      Rs[(size_t)comp * S + l] = ru;
      Rs[(size_t)(comp + 6) * S + l] = rl;
    }
    // the next step reads neighbours' r; the last one's barrier keeps every CTA until the others have
    // read its sites
    if (CLS > 1) cluster.sync();
    else __syncthreads();
  }
  if (active) {
    pz[(size_t)comp * V + x] = pz[(size_t)comp * V + x] + xu;
    pz[(size_t)(comp + 6) * V + x] = pz[(size_t)(comp + 6) * V + x] + xl;
  }
}

// CTAs per block: at most 64 sites (384 threads, 64 KB of shared memory: two or three CTAs per SM) where a
// cluster of eight reaches that, and more CTAs as long as there are fewer than SMs and a CTA keeps 16
// sites.  The rule looks at the level only, not at the batch: the partial sums of a block must not
// depend on it.
int split_ctas(int vB, int nblocks) {
  int CLS = 1;
  while (CLS < MAXCLS && (vB > 64 * CLS || (nblocks * CLS < SMS && vB >= 32 * CLS))) CLS *= 2;
  return CLS;
}

}  // namespace

namespace dd {

void fine_dslash_split(cplx<double>* out, const cplx<double>* in, const cplx<double>* b, const FineOp<double>& op,
                       int nrhs, size_t rstride, cudaStream_t st) {
  const dim3 grid(div_up(op.g.V, DS), nrhs);
  count_launch();
  if (b)
    k_fine_dslash_split<true><<<grid, 6 * DS, 0, st>>>(out, in, b, op.U, op.clov, op.g, op.bc_t, rstride);
  else
    k_fine_dslash_split<false><<<grid, 6 * DS, 0, st>>>(out, in, b, op.U, op.clov, op.g, op.bc_t, rstride);
}

// Six threads per site against one (k_fine_sap, CTAs of 256 threads).  With one, a wave of 152 CTAs takes 34 us and 47 for
// each warp of a CTA that has sites, however few CTAs run.  Six take, for the sites of the SM with the most CTAs, 0.81 us
// per site and 0.15 for each hop pass of an MR step (3 MR steps).  So six threads lose where the blocks of a
// colour, for all right-hand sides, fill the waves of the other kernel.  us per sweep, six / one: 4^4 blocks, 32: 139 / 405,
// 96: 378 / 403, 128: 490 / 404, 192: 690 / 800, 256: 916 / 800, 768: 2518 / 2380; 4^3 x 2, 256: 442 / 400, 384: 622 / 790;
// 4^2 x 2^2, 512 in one field: 459 / 413, 128 in four: 377 / 405; 3^3 x 2, 2304: 1727 / 1638; 3^4, 128: 168 / 318,
// 512: 561 / 630; 2^4, 2048: 325 / 410.
// Above 256 sites one thread per site takes more registers than a CTA has.  The two sum in different orders and a column has
// the same bits alone and in a batch, so the rule counts the batch that the handle was set up for, not the one at
// hand.  With 16 4^4 blocks a handle for one right-hand side smooths eight fields in 62 us each instead of 50, and a handle for
// eight smooths one in 408 us instead of 135.
bool fine_sap_takes_split(const Geom& g, int nblocks, int batch) {
  const int vB = g.vB, CLS = split_ctas(vB, nblocks), S = (vB + CLS - 1) / CLS;
  if (vB > 256) return true;
  int passes = 0, seg = 1;
  for (int d = 0; d < 4; ++d) passes += g.B[d] == g.L[d] || g.B[d] > 2 ? 2 : g.B[d] - 1;
  while (seg < vB) seg <<= 1;
  const int per_cta = 256 / seg, warps = seg >= 32 ? per_cta * ((vB + 31) / 32) : 8;
  const long long blocks = (long long)nblocks * batch;
  auto waves = [](long long ctas) { return (double)((ctas + SMS - 1) / SMS); };
  const double one = waves((blocks + per_cta - 1) / per_cta) * (34.0 + 47.0 * warps);
  const double sites = (6 * S + 31) / 32 * 32 / 6.0;   // of a CTA, with the threads that have none
  return waves(blocks * CLS) * sites * (0.81 + 0.15 * passes) < one;
}

cudaError_t fine_sap_split(cplx<double>* z, const cplx<double>* b, const FineOp<double>& op, const int* blocks,
                           int nblocks, int nrhs, size_t rstride, int k_mr, cudaStream_t st) {
  if (k_mr < 1) return cudaSuccess;   // e = 0
  const int vB = op.g.vB;
  const int CLS = split_ctas(vB, nblocks);
  const int S = (vB + CLS - 1) / CLS;
  const int threads = ((6 * S + 31) / 32) * 32;
  const size_t sm = (size_t)66 * S * sizeof(cplx<double>) + (72 + 6 * MAXCLS) * sizeof(double) + (size_t)8 * S * sizeof(short);
  if (threads > 768 || sm > 227 * 1024) return cudaErrorInvalidConfiguration;
  static DeviceOnce once384, once768;
  if (threads <= 384) raise_smem_limit(once384, (const void*)k_fine_sap_split<384>);
  else raise_smem_limit(once768, (const void*)k_fine_sap_split<768>);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CLS;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(nblocks * CLS, nrhs, 1);
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  count_launch();
  return cudaLaunchKernelEx(&cfg, threads <= 384 ? k_fine_sap_split<384> : k_fine_sap_split<768>, z, b, (const cplx<double>*)op.U, (const double*)op.clov, op.g,
                            op.bc_t, rstride, blocks, k_mr, S);
}

}  // namespace dd
