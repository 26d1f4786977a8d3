// Batched BLAS-1 and the per-right-hand-side GMRES bookkeeping.
//
// Reductions are deterministic and independent of the batch: every rhs is
// reduced over the same fixed partition of its vector (stage 1: one partial
// per CTA-chunk, stage 2: one CTA sums the partials in a fixed order), so a
// right-hand side gives bit-identical results alone or inside a batch.
#include "common.cuh"
#include "kernels.h"

#include <stdexcept>
#include <type_traits>
#include <unordered_map>

#include <cstdio>
#include <atomic>
#include <mutex>

namespace {

constexpr int RT = 256;         // threads per reduction CTA
constexpr int MAXCHUNKS = 512;  // partials per rhs (and per dot in a multidot)

// scratch for the partials, one buffer per stream (reductions issued on different streams, as by
// the serving workers of several hierarchies, never share scratch), grown on demand
// (library-owned device memory).  A buffer that was replaced is kept until the library is
// unloaded, because captured CUDA graphs may still refer to it.
struct PartialBuf {
  double* p = nullptr;
  size_t cap = 0;
};
std::mutex g_partials_mu;
std::unordered_map<cudaStream_t, PartialBuf> g_partials;

double* partials(size_t count, cudaStream_t st) {
  std::lock_guard<std::mutex> lk(g_partials_mu);
  PartialBuf& b = g_partials[st];
  if (count > b.cap) {
    const size_t cap = count < (1u << 17) ? (1u << 17) : count;
    double* p = nullptr;
    if (cudaMalloc(&p, cap * sizeof(double)) != cudaSuccess) {
      cudaGetLastError();
      throw std::runtime_error("out of device memory for reduction partials");
    }
    b.p = p;
    b.cap = cap;
  }
  return b.p;
}

int nchunks(size_t len) {
  size_t c = (len + 2 * RT - 1) / (2 * RT);
  if (c < 1) c = 1;
  if (c > MAXCHUNKS) c = MAXCHUNKS;
  return (int)c;
}

__device__ double warp_sum(double v) {
  for (int off = 16; off >= 1; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// sum `cnt` doubles per thread over the CTA (cnt <= 8); thread 0 gets the result
__device__ void cta_sum(double* v, int cnt, double* sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int k = 0; k < cnt; ++k) v[k] = warp_sum(v[k]);
  if (lane == 0)
    for (int k = 0; k < cnt; ++k) sh[warp * 8 + k] = v[k];
  __syncthreads();
  if (threadIdx.x == 0)
    for (int k = 0; k < cnt; ++k) {
      double s = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += sh[w * 8 + k];
      v[k] = s;
    }
  __syncthreads();
}

// chunk [lo, hi) of a vector of length len split into nc chunks
__device__ void chunk_range(size_t len, int nc, int c, size_t& lo, size_t& hi) {
  const size_t per = (len + nc - 1) / nc;
  lo = (size_t)c * per;
  hi = lo + per;
  if (hi > len) hi = len;
  if (lo > len) lo = len;
}

// Sum 8 values per thread over the CTA (RT threads); thread k < 8 returns the sum of value k.  The lanes share the
// values out as they fold (9 additions per lane), and eight threads add the warps' sums.  The order is that of
// a butterfly over the lanes, then the warps by number.
__device__ __forceinline__ double cta_fold8(double* v, double* sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int w = 4, off = 16; w >= 1; w >>= 1, off >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int k = 0; k < w; ++k) {
      const double keep = up ? v[k + w] : v[k], send = up ? v[k] : v[k + w];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
  if ((lane & 3) == 0) sh[warp * 8 + (lane >> 2)] = v[0];
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x < 8)
#pragma unroll
    for (int w = 0; w < RT / 32; ++w) s += sh[w * 8 + threadIdx.x];
  return s;
}

// Stage 1 of dot: partial[(rhs * m + d) * nc + chunk] (re, im); blockIdx.z = group of four vectors d.
// Bound by the FP64 rate, at FP32 by the launch: with the groups in one CTA one after another, 40 additions per lane
// and group for the CTA sum and 48 CTAs for 8^4, 13 vectors of 8^4 took 51 us and six of 16^3x32 114 us.  Now 12
// and 76 us (the FP64 rate: 72).
template <typename T>
__global__ void __launch_bounds__(RT) k_multidot1(double* __restrict__ part, const cplx<T>* __restrict__ V,
                                                  size_t vstride, int m, const cplx<T>* __restrict__ w, size_t len,
                                                  size_t rstride, int nc) {
  __shared__ double sh[RT / 32 * 8];
  const int chunk = blockIdx.x, rhs = blockIdx.y, d0 = 4 * blockIdx.z, nd = min(4, m - d0);
  size_t lo, hi;
  chunk_range(len, nc, chunk, lo, hi);
  const cplx<T>* pw = w + (size_t)rhs * rstride;
  const cplx<T>* pv = V + (size_t)d0 * vstride + (size_t)rhs * rstride;
  // per-thread partials in the precision of the data (FP32 data: FP32 sums)
  T at[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  auto products = [&](auto count) {   // a skipped FP64 FMA takes its time all the same: a loop for each count
    for (size_t e = lo + threadIdx.x; e < hi; e += RT) {
      const cplx<T> we = pw[e];
#pragma unroll
      for (int dd = 0; dd < decltype(count)::value; ++dd)
        cdotc_acc(at[2 * dd], at[2 * dd + 1], pv[(size_t)dd * vstride + e], we);
    }
  };
  if (nd == 4) products(std::integral_constant<int, 4>());
  else if (nd == 3) products(std::integral_constant<int, 3>());
  else if (nd == 2) products(std::integral_constant<int, 2>());
  else products(std::integral_constant<int, 1>());
  double acc[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) acc[k] = (double)at[k];
  const double t = cta_fold8(acc, sh);
  if (threadIdx.x < 2 * nd)
    part[(((size_t)rhs * m + d0 + (threadIdx.x >> 1)) * nc + chunk) * 2 + (threadIdx.x & 1)] = t;
}

// stage 1 of the multidot in double-FP32 arithmetic on FP64 vectors: the elements are split on
// load, products and the per-thread sums are double-FP32, the CTA sum is FP64 (partials as above)
__global__ void __launch_bounds__(RT) k_multidot1_df(double* __restrict__ part, const cplx<double>* __restrict__ V,
                                                     size_t vstride, int m, const cplx<double>* __restrict__ w,
                                                     size_t len, size_t rstride, int nc) {
  __shared__ double sh[RT / 32 * 8];
  const int chunk = blockIdx.x, rhs = blockIdx.y, d0 = 4 * blockIdx.z, nd = min(4, m - d0);
  size_t lo, hi;
  chunk_range(len, nc, chunk, lo, hi);
  const cplx<double>* pw = w + (size_t)rhs * rstride;
  const cplx<double>* pv = V + (size_t)d0 * vstride + (size_t)rhs * rstride;
  dfl at[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) at[k] = dfl(0);
  for (size_t e = lo + threadIdx.x; e < hi; e += RT) {
    const cplx<double> wd = pw[e];
    const dfl wr = df_from_double(wd.re), wi = df_from_double(wd.im);
#pragma unroll
    for (int dd = 0; dd < 4; ++dd) {
      if (dd < nd) {
        const cplx<double> vd = pv[(size_t)dd * vstride + e];
        const dfl vr = df_from_double(vd.re), vi = df_from_double(vd.im);
        // conj(v) w
        at[2 * dd] = fma(vr, wr, at[2 * dd]);
        at[2 * dd] = fma(vi, wi, at[2 * dd]);
        at[2 * dd + 1] = fma(vr, wi, at[2 * dd + 1]);
        at[2 * dd + 1] = fma(-vi, wr, at[2 * dd + 1]);
      }
    }
  }
  double acc[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) acc[k] = df_to_double(at[k]);
  const double t = cta_fold8(acc, sh);
  if (threadIdx.x < 2 * nd)
    part[(((size_t)rhs * m + d0 + (threadIdx.x >> 1)) * nc + chunk) * 2 + (threadIdx.x & 1)] = t;
}

// stage 2: res[rhs * m + d] = sum over chunks, fixed order
__global__ void k_multidot2(cplx<double>* __restrict__ res, const double* __restrict__ part, int m, int nc,
                            int res_stride) {
  __shared__ double sh[32 * 8];
  const int d = blockIdx.x, rhs = blockIdx.y;
  const double* p = part + ((size_t)rhs * m + d) * nc * 2;
  double acc[2] = {0.0, 0.0};
  for (int c = threadIdx.x; c < nc; c += blockDim.x) { acc[0] += p[2 * c]; acc[1] += p[2 * c + 1]; }
  cta_sum(acc, 2, sh);
  if (threadIdx.x == 0) res[(size_t)rhs * res_stride + d] = cmk(acc[0], acc[1]);
}

template <typename T>
__global__ void k_norm1(double* __restrict__ part, const cplx<T>* __restrict__ x, size_t len, size_t rstride, int nc) {
  __shared__ double sh[32 * 8];
  const int chunk = blockIdx.x, rhs = blockIdx.y;
  size_t lo, hi;
  chunk_range(len, nc, chunk, lo, hi);
  const cplx<T>* px = x + (size_t)rhs * rstride;
  T at = T(0);
  for (size_t e = lo + threadIdx.x; e < hi; e += blockDim.x) {
    const cplx<T> v = px[e];
    cnorm2_acc(at, v);
  }
  double acc[1] = {(double)at};
  cta_sum(acc, 1, sh);
  if (threadIdx.x == 0) part[(size_t)rhs * nc + chunk] = acc[0];
}

__global__ void k_norm2(double* __restrict__ res, const double* __restrict__ part, int nc) {
  __shared__ double sh[32 * 8];
  const int rhs = blockIdx.x;
  double acc[1] = {0.0};
  for (int c = threadIdx.x; c < nc; c += blockDim.x) acc[0] += part[(size_t)rhs * nc + c];
  cta_sum(acc, 1, sh);
  if (threadIdx.x == 0) res[rhs] = sqrt(acc[0]);
}

template <typename T>
__global__ void k_multiaxpy(cplx<T>* __restrict__ y, const cplx<T>* __restrict__ V, size_t vstride, int m,
                            const cplx<double>* __restrict__ c, int cstride, double sign, size_t len,
                            size_t rstride) {
  // coefficients sign * c_i of this right-hand side, computed once per CTA; a zero
  // coefficient skips its vector (never touch unused, possibly unset vectors)
  __shared__ cplx<T> cs[64];
  __shared__ int use[64];
  const int rhs = blockIdx.y;
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    const cplx<double> ci = c[(size_t)rhs * cstride + i];
    use[i] = !(ci.re == 0.0 && ci.im == 0.0);
    cs[i] = cmk<T>((T)(sign * ci.re), (T)(sign * ci.im));
  }
  __syncthreads();
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= len) return;
  const size_t o = (size_t)rhs * rstride + e;
  cplx<T> acc = y[o];
  for (int i = 0; i < m; ++i) {
    if (!use[i]) continue;
    cfma(acc, cs[i], V[(size_t)i * vstride + o]);
  }
  y[o] = acc;
}

// y += sign * sum_i c_i V_i in double-FP32 arithmetic on FP64 vectors (result rounded to FP64)
__global__ void k_multiaxpy_df(cplx<double>* __restrict__ y, const cplx<double>* __restrict__ V, size_t vstride,
                               int m, const cplx<double>* __restrict__ c, int cstride, double sign, size_t len,
                               size_t rstride) {
  __shared__ cplx<dfl> cs[64];
  __shared__ int use[64];
  const int rhs = blockIdx.y;
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    const cplx<double> ci = c[(size_t)rhs * cstride + i];
    use[i] = !(ci.re == 0.0 && ci.im == 0.0);
    const double a = sign * ci.re, b = sign * ci.im;
    const float ah = __double2float_rn(a), bh = __double2float_rn(b);
    cs[i] = cmk<dfl>(dfl(ah, __double2float_rn(a - (double)ah)), dfl(bh, __double2float_rn(b - (double)bh)));
  }
  __syncthreads();
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= len) return;
  const size_t o = (size_t)rhs * rstride + e;
  const cplx<double> yd = y[o];
  cplx<dfl> acc = cmk<dfl>(df_from_double(yd.re), df_from_double(yd.im));
  for (int i = 0; i < m; ++i) {
    if (!use[i]) continue;
    const cplx<double> vd = V[(size_t)i * vstride + o];
    cfma(acc, cs[i], cmk<dfl>(df_from_double(vd.re), df_from_double(vd.im)));
  }
  y[o] = cmk<double>(df_to_double(acc.re), df_to_double(acc.im));
}

template <typename T>
__global__ void k_scale_to(cplx<T>* y, const cplx<T>* x, const double* __restrict__ a,
                           size_t len, size_t rstride) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= len) return;
  const size_t o = (size_t)blockIdx.y * rstride + e;
  const T s = (T)a[blockIdx.y];
  y[o] = s * x[o];
}

template <typename T>
__global__ void k_axpy(cplx<T>* __restrict__ y, const cplx<T>* __restrict__ x, double a, size_t len, size_t rstride) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= len) return;
  const size_t o = (size_t)blockIdx.y * rstride + e;
  y[o] = y[o] + (T)a * x[o];
}

template <typename To, typename Ti>
__global__ void k_convert(cplx<To>* y, const cplx<Ti>* x, size_t len, size_t ys, size_t xs) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= len) return;
  y[(size_t)blockIdx.y * ys + e] = ccast<To>(x[(size_t)blockIdx.y * xs + e]);
}

template <typename T>
__global__ void k_zero(cplx<T>* __restrict__ y, size_t len, size_t rstride) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= len) return;
  y[(size_t)blockIdx.y * rstride + e] = czero<T>();
}

__global__ void k_recip(double* __restrict__ a, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) a[i] = a[i] > 0.0 ? 1.0 / a[i] : 0.0;
}

template <typename T>
__global__ void k_real_convert(T* __restrict__ y, const double* __restrict__ x, size_t len) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < len) y[e] = (T)x[e];
}

// ---- GMRES (one thread per rhs) ----------------------------------------------
// Givens convention: [[c, s], [-conj(s), c]] (a, b)^T = (rho, 0)^T with c real.
__device__ void givens(cplx<double> a, cplx<double> b, double& c, cplx<double>& s) {
  const double aa = sqrt(cnorm2(a)), bb = sqrt(cnorm2(b));
  const double r = hypot(aa, bb);
  if (r == 0.0) { c = 1.0; s = czero<double>(); return; }
  if (aa == 0.0) { c = 0.0; s = bb == 0.0 ? cmk(1.0, 0.0) : cmk(b.re / bb, -b.im / bb); return; }
  c = aa / r;
  const cplx<double> ph = cmk(a.re / aa, a.im / aa);
  s = (1.0 / r) * (ph * cconj(b));
}

__global__ void k_gmres_begin(dd::GmresState s, int nrhs) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= nrhs) return;
  const int m = s.m;
  for (int k = 0; k <= m; ++k) s.g[(size_t)r * (m + 1) + k] = czero<double>();
  const double b = s.beta[r];
  s.g[(size_t)r * (m + 1)] = cmk(b, 0.0);
  s.kr[r] = 0;
  s.done[r] = (b <= s.target[r]) ? 1 : 0;
  s.inv[r] = (b > 0.0 && !s.done[r]) ? 1.0 / b : 0.0;
  s.est[r] = b;
}

// One Arnoldi column per right-hand side: a warp each.  The j rotations of the earlier steps are a chain in the
// running entry alone: lane 0 carries its real part and lane 1 its imaginary part (two FP64 FMAs and a shuffle per
// rotation), what does not depend on it is formed by all lanes before and after.  8^4, steps 0 to 25:
// 9.8 us on average (15.2 by one thread, whose FP64 operations take 31 ns each).
__global__ void __launch_bounds__(32) k_gmres_step(dd::GmresState s, int j) {
  __shared__ cplx<double> hh[65], cur[65], sh_sn[64];
  __shared__ double sh_cs[64];
  const int r = blockIdx.x, lane = threadIdx.x;
  if (s.done[r]) {   // finished rhs: next basis vector is exactly zero
    if (lane == 0) s.inv[r] = 0.0;
    return;
  }
  const int m = s.m;
  cplx<double>* H = s.H + (size_t)r * (m + 1) * m;
  cplx<double>* g = s.g + (size_t)r * (m + 1);
  double* cs = s.cs + (size_t)r * m;
  cplx<double>* sn = s.sn + (size_t)r * m;
  const double hn = s.wnorm[r];
  for (int i = lane; i <= j; i += 32) {
    hh[i] = s.h1[(size_t)r * (m + 1) + i] + s.h2[(size_t)r * (m + 1) + i];
    if (i < j) {
      sh_cs[i] = cs[i];
      sh_sn[i] = sn[i];
    }
  }
  __syncwarp();
  for (int i = lane; i < j; i += 32) cur[i + 1] = sh_cs[i] * hh[i + 1];
  __syncwarp();
  if (lane == 0) cur[0] = hh[0];
  __syncwarp();
  if (j > 0) {
    const int p = lane & 1;   // every lane computes; lanes 0 and 1 store
    double c = p ? cur[0].im : cur[0].re;
    for (int i = 0; i < j; ++i) {
      const cplx<double> si = sh_sn[i];
      const double a = p ? cur[i + 1].im : cur[i + 1].re, im = p ? si.im : -si.im;
      const double o = __shfl_xor_sync(0xffffffffu, c, 1);
      c = fma(im, o, fma(-si.re, c, a));   // cs h_{i+1} - conj(sn) h_i
      __syncwarp();
      if (lane < 2) reinterpret_cast<double*>(&cur[i + 1])[p] = c;
    }
  }
  __syncwarp();
  for (int i = lane; i < j; i += 32) H[(size_t)i * m + j] = sh_cs[i] * cur[i] + sh_sn[i] * hh[i + 1];
  if (lane) return;
  const cplx<double> h0 = cur[j], h1 = cmk(hn, 0.0);
  double c;
  cplx<double> sg;
  givens(h0, h1, c, sg);
  cs[j] = c;
  sn[j] = sg;
  H[(size_t)j * m + j] = c * h0 + sg * h1;
  H[(size_t)(j + 1) * m + j] = czero<double>();
  const cplx<double> gj = g[j], g1 = -1.0 * (cconj(sg) * gj);
  g[j + 1] = g1;
  g[j] = c * gj;
  s.kr[r] = j + 1;
  const double est = sqrt(cnorm2(g1));
  s.est[r] = est;
  s.inv[r] = hn > 0.0 ? 1.0 / hn : 0.0;
  if (est <= s.target[r] || hn == 0.0 || j + 1 == m) { s.done[r] = 1; s.inv[r] = 0.0; }
}

// y = R^{-1} g, a warp per right-hand side: R's upper triangle by columns in shared memory; with y_i known, all
// lanes subtract its column from the rows above.
__global__ void __launch_bounds__(32) k_gmres_solve_y(dd::GmresState s) {
  __shared__ cplx<double> R[64 * 63 / 2];   // above the diagonal: column l from l (l - 1) / 2
  __shared__ cplx<double> t[64], id[64];
  const int r = blockIdx.x, lane = threadIdx.x;
  const int m = s.m;
  const int k = s.kr[r];
  const cplx<double>* H = s.H + (size_t)r * (m + 1) * m;
  const cplx<double>* g = s.g + (size_t)r * (m + 1);
  cplx<double>* y = s.y + (size_t)r * m;
  for (int i = k + lane; i < m; i += 32) y[i] = czero<double>();
  for (int i = 0; i < k; ++i)
    for (int l = i + 1 + lane; l < k; l += 32) R[l * (l - 1) / 2 + i] = H[(size_t)i * m + l];
  for (int i = lane; i < k; i += 32) {
    const cplx<double> d = H[(size_t)i * m + i];
    const double dn = cnorm2(d);
    id[i] = dn > 0.0 ? (1.0 / dn) * cconj(d) : czero<double>();
    t[i] = g[i];
  }
  __syncwarp();
  for (int i = k - 1; i >= 0; --i) {
    const cplx<double> yi = t[i] * id[i];
    for (int l = lane; l < i; l += 32) t[l] = t[l] - R[i * (i - 1) / 2 + l] * yi;
    if (lane == 0) y[i] = yi;
    __syncwarp();
  }
}

}  // namespace

namespace dd {

static std::atomic<long long> g_launches{0};
void count_launch(int k) { g_launches.fetch_add(k, std::memory_order_relaxed); }
long long launch_count() { return g_launches.load(std::memory_order_relaxed); }

template <typename T>
void blas_multidot(cplx<double>* res, int res_stride, const cplx<T>* V, size_t vstride, int m, const cplx<T>* w,
                   size_t len, int nrhs, size_t rstride, cudaStream_t st) {
  if (m <= 0) return;
  const int nc = nchunks(len);
  double* part = partials((size_t)nrhs * m * nc * 2, st);
  count_launch();
  k_multidot1<T><<<dim3(nc, nrhs, div_up(m, 4)), RT, 0, st>>>(part, V, vstride, m, w, len, rstride, nc);
  count_launch();
  k_multidot2<<<dim3(m, nrhs), 128, 0, st>>>(res, part, m, nc, res_stride);
}

void blas_multidot_df(cplx<double>* res, int res_stride, const cplx<double>* V, size_t vstride, int m,
                      const cplx<double>* w, size_t len, int nrhs, size_t rstride, cudaStream_t st) {
  if (m <= 0) return;
  const int nc = nchunks(len);
  double* part = partials((size_t)nrhs * m * nc * 2, st);
  count_launch();
  k_multidot1_df<<<dim3(nc, nrhs, div_up(m, 4)), RT, 0, st>>>(part, V, vstride, m, w, len, rstride, nc);
  count_launch();
  k_multidot2<<<dim3(m, nrhs), 128, 0, st>>>(res, part, m, nc, res_stride);
}

void blas_multiaxpy_df(cplx<double>* y, const cplx<double>* V, size_t vstride, int m, const cplx<double>* c,
                       int cstride, double sign, size_t len, int nrhs, size_t rstride, cudaStream_t st) {
  if (m <= 0) return;
  if (m > 64) throw std::runtime_error("blas_multiaxpy_df: at most 64 vectors");
  count_launch();
  k_multiaxpy_df<<<dim3(div_up(len, 256), nrhs), 256, 0, st>>>(y, V, vstride, m, c, cstride, sign, len, rstride);
}

void reserve_partials(int nrhs, int m, cudaStream_t st) { partials((size_t)nrhs * (m + 1) * MAXCHUNKS * 2, st); }

template <typename T>
void blas_dot(cplx<double>* res, const cplx<T>* x, const cplx<T>* y, size_t len, int nrhs, size_t rstride,
              cudaStream_t st) {
  blas_multidot<T>(res, 1, x, 0, 1, y, len, nrhs, rstride, st);
}

template <typename T>
void blas_norm2(double* res, const cplx<T>* x, size_t len, int nrhs, size_t rstride, cudaStream_t st) {
  const int nc = nchunks(len);
  double* part = partials((size_t)nrhs * nc, st);
  count_launch();
  k_norm1<T><<<dim3(nc, nrhs), RT, 0, st>>>(part, x, len, rstride, nc);
  count_launch();
  k_norm2<<<nrhs, 128, 0, st>>>(res, part, nc);
}

template <typename T>
void blas_multiaxpy(cplx<T>* y, const cplx<T>* V, size_t vstride, int m, const cplx<double>* c, int cstride,
                    double sign, size_t len, int nrhs, size_t rstride, cudaStream_t st) {
  if (m <= 0) return;
  if (m > 64) throw std::runtime_error("blas_multiaxpy: at most 64 vectors");
  count_launch();
  k_multiaxpy<T><<<dim3(div_up(len, 256), nrhs), 256, 0, st>>>(y, V, vstride, m, c, cstride, sign, len, rstride);
}

template <typename T>
void blas_scale_to(cplx<T>* y, const cplx<T>* x, const double* a, size_t len, int nrhs, size_t rstride,
                   cudaStream_t st) {
  count_launch();
  k_scale_to<T><<<dim3(div_up(len, 256), nrhs), 256, 0, st>>>(y, x, a, len, rstride);
}

template <typename T>
void blas_axpy(cplx<T>* y, const cplx<T>* x, double a, size_t len, int nrhs, size_t rstride, cudaStream_t st) {
  count_launch();
  k_axpy<T><<<dim3(div_up(len, 256), nrhs), 256, 0, st>>>(y, x, a, len, rstride);
}

template <typename To, typename Ti>
void blas_convert(cplx<To>* y, const cplx<Ti>* x, size_t len, int nrhs, size_t ystride, size_t xstride,
                  cudaStream_t st) {
  count_launch();
  k_convert<To, Ti><<<dim3(div_up(len, 256), nrhs), 256, 0, st>>>(y, x, len, ystride, xstride);
}

template <typename T>
void blas_zero(cplx<T>* y, size_t len, int nrhs, size_t rstride, cudaStream_t st) {
  count_launch();
  k_zero<T><<<dim3(div_up(len, 256), nrhs), 256, 0, st>>>(y, len, rstride);
}

template <typename T>
void real_convert(T* y, const double* x, size_t len, cudaStream_t st) {
  count_launch();
  k_real_convert<T><<<div_up(len, 256), 256, 0, st>>>(y, x, len);
}

void blas_recip(double* a, int n, cudaStream_t st) { k_recip<<<div_up(n, 128), 128, 0, st>>>(a, n); }

void gmres_begin(const GmresState& s, int nrhs, cudaStream_t st) { k_gmres_begin<<<div_up(nrhs, 32), 32, 0, st>>>(s, nrhs); }
void gmres_step(const GmresState& s, int j, int nrhs, cudaStream_t st) {
  count_launch();
  k_gmres_step<<<nrhs, 32, 0, st>>>(s, j);
}
void gmres_solve_y(const GmresState& s, int nrhs, cudaStream_t st) {
  count_launch();
  k_gmres_solve_y<<<nrhs, 32, 0, st>>>(s);
}

#define INST(T)                                                                                                 \
  template void blas_multidot<T>(cplx<double>*, int, const cplx<T>*, size_t, int, const cplx<T>*, size_t, int,   \
                                 size_t, cudaStream_t);                                                         \
  template void blas_dot<T>(cplx<double>*, const cplx<T>*, const cplx<T>*, size_t, int, size_t, cudaStream_t);   \
  template void blas_norm2<T>(double*, const cplx<T>*, size_t, int, size_t, cudaStream_t);                      \
  template void blas_multiaxpy<T>(cplx<T>*, const cplx<T>*, size_t, int, const cplx<double>*, int, double,      \
                                  size_t, int, size_t, cudaStream_t);                                           \
  template void blas_scale_to<T>(cplx<T>*, const cplx<T>*, const double*, size_t, int, size_t, cudaStream_t);   \
  template void blas_axpy<T>(cplx<T>*, const cplx<T>*, double, size_t, int, size_t, cudaStream_t);              \
  template void blas_zero<T>(cplx<T>*, size_t, int, size_t, cudaStream_t);                                      \
  template void real_convert<T>(T*, const double*, size_t, cudaStream_t);
INST(float)
INST(double)
#undef INST
template void blas_convert<float, double>(cplx<float>*, const cplx<double>*, size_t, int, size_t, size_t, cudaStream_t);
template void blas_convert<double, float>(cplx<double>*, const cplx<float>*, size_t, int, size_t, size_t, cudaStream_t);
template void blas_convert<double, double>(cplx<double>*, const cplx<double>*, size_t, int, size_t, size_t,
                                           cudaStream_t);
template void blas_convert<float, float>(cplx<float>*, const cplx<float>*, size_t, int, size_t, size_t, cudaStream_t);

}  // namespace dd
