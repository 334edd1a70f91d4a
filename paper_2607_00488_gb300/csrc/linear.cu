// Exact rank-8 evaluation of the likelihood (srw_loglik_linear in srw.h).
//
// The recoil spectrum is a polynomial in the shifted couplings and mu_hat^2
// (Sec. II: eqs. sm_cross_section, g_tilde, xs_mm, xs_total), so the weighted
// true spectrum is W(theta) = sum_b c_b(theta) shat_b with eight fixed
// coefficient spectra, and the fold of eq. matrix_reweight is linear in them:
//
//   mu(theta) = R W_ref + b + M (c(theta) - c_ref),   M = R shat^T  [n_rec][8]
//
// M is computed once in FP64 (per rec bin, eight dot products of length n_t).
// Per point the kernel forms the eight coefficients, then per rec bin
// Delta = sum_b M_jb (c_b - c_ref,b) (8 FMAs), mu = mu_ref + b + Delta, and the
// Poisson deviance of eq. logL from d = n - mu and s = n + mu (the same series
// / log forms as the batched epilogues), accumulated in double-float.  The
// same linearity gives the gradient:
//   d(-2 ln L)/d theta_k = 2 sum_b (d c_b / d theta_k) sum_j M_jb (1 - n_j/mu_j).
// Four threads per point, each on every fourth rec bin, in four warps: all
// lanes of a warp are at the same bin, so that the branches below are taken by
// whole warps.  The per-bin constants are staged through shared memory and
// read as broadcasts.
//
// What bounds both kernels: instruction issue.  With four adjacent lanes per
// point every term paid for the series and the logarithm (bins with few counts,
// which need the logarithm, lie beside bins that do not): 67 instructions a
// term.  At one bin per warp a bin without data is one addition (t = mu), the
// form that no point of the warp needs is left out, and a thread with two
// points forms both in packed FP32 instructions and shares the loads.

#include "dfloat.cuh"
#include "f32x2.cuh"
#include "poisson.cuh"
#include "srw_internal.h"

namespace srw {
namespace {

constexpr int kLinThreads = 128;              // a warp per residue of the rec bin modulo 4
constexpr int kLinChunk = 256;                // rec bins per shared-memory chunk
constexpr int kSplitThreads = 512;            // split kernels (few points): sixteen warps on a round of
constexpr int kSplitRound = 64;               // 64 rec bins
constexpr int kSplitChunk = 1024;             // 48 KB of constants beside 16 KB of terms (L = 8; 32 KB at L = 16)
constexpr int kProfChunk = 2048;              // 96 KB of constants, staged once up to this many bins

// M_jb = sum_i R_ji shat_b,i with shat_b,i = B_b,i E_SM,i / S_SM,i (FP64); one
// block per rec bin.
__global__ void linear_m_kernel(const float* __restrict__ R, int ld, int n_t, const double* __restrict__ basis,
                                const double* __restrict__ ssm, const double* __restrict__ esm, double* __restrict__ M) {
  __shared__ double red[kNB][32];
  const int j = blockIdx.x;
  double acc[kNB];
#pragma unroll
  for (int b = 0; b < kNB; ++b) acc[b] = 0.0;
  for (int i = threadIdx.x; i < n_t; i += blockDim.x) {
    const double r = (double)R[(size_t)j * ld + i];
    if (r == 0.0) continue;
    const double sm = ssm[i], e = esm[i];
#pragma unroll
    for (int b = 0; b < kNB; ++b) {
      const double sh = sm != 0.0 ? basis[(size_t)b * n_t + i] * (e / sm) : (b == 6 ? e : 0.0);
      acc[b] += r * sh;
    }
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int b = 0; b < kNB; ++b) {
    double v = acc[b];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[b][w] = v;
  }
  __syncthreads();
  if (threadIdx.x < kNB) {
    double t = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += red[threadIdx.x][k];
    M[(size_t)j * kNB + threadIdx.x] = t;
  }
}

// Per-bin constants: {M_j0..3}, {M_j4, M_j5, M_j7, n - mu_ref - b}, {n + mu_ref + b, n, mask, 0} (the
// constant monomial's deviation is always zero), and for the profiled evaluation {mu_ref, b, n (or -1: masked), 0}.
__global__ void linear_consts_kernel(const double* __restrict__ M, const double* __restrict__ n64,
                                     const double* __restrict__ bref64, const double* __restrict__ muref,
                                     const unsigned char* __restrict__ mask, int n_rec, float4* __restrict__ out,
                                     float4* __restrict__ outp) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n_rec) return;
  const double* m = M + (size_t)j * kNB;
  const double n = n64[j], base = bref64[j];
  const bool on = mask == nullptr || mask[j] != 0;
  // masked bins: n = 0; a count below FP32's quotients is the smallest that has data
  const double nn = !on || n == 0.0 ? 0.0 : fmax(n, 1e-30);
  out[3 * j] = make_float4((float)m[0], (float)m[1], (float)m[2], (float)m[3]);
  out[3 * j + 1] = make_float4((float)m[4], (float)m[5], (float)m[7], (float)(nn - base));
  out[3 * j + 2] = make_float4((float)(nn + base), (float)nn, on ? 1.f : 0.f, 0.f);
  outp[j] = make_float4((float)muref[j], (float)(base - muref[j]), on ? (float)nn : -1.f, 0.f);
}

struct Couplings {
  float gle, gre, glt, grt, mu;
};

__device__ __forceinline__ void deviations(const float* th, dfloat s, const CoefRef& ref, float* c, Couplings& g) {
  const dfloat gle = df_add(df_add(dfloat{0.5f, 0.f}, s), th[0]), gre = df_add(s, th[1]);
  const dfloat glt = df_add(df_add(dfloat{-0.5f, 0.f}, s), th[2]), grt = df_add(s, th[3]);
  const dfloat x = df_mul(gle, gre), y = df_mul(glt, grt);
  const dfloat v[kNB] = {df_mul(gle, gle), df_mul(gre, gre), {-x.hi, -x.lo}, df_mul(glt, glt),
                         df_mul(grt, grt), {-y.hi, -y.lo}, {1.f, 0.f}, two_prod(th[4], th[4])};
#pragma unroll
  for (int b = 0; b < kNB; ++b) {
    const dfloat d = df_add(v[b], dfloat{-ref.hi[b], -ref.lo[b]});
    c[b] = d.hi + d.lo;
  }
  g = Couplings{gle.hi + gle.lo, gre.hi + gre.lo, glt.hi + glt.lo, grt.hi + grt.lo, th[4]};
}

// n / mu of N points in a bin with data.  A tiny mu takes CUDA's fast division
// instead, and only that quotient does: which other points and bins share a warp
// does not touch a value.
template <int N>
__device__ __forceinline__ void quotients(float n, const float* mu, float* q) {
  bool fine = true;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    q[i] = quotient(n, mu[i]);
    fine = fine && !(fabsf(mu[i]) < 1e-30f);
  }
  if (!__all_sync(0xffffffffu, fine)) {
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (fabsf(mu[i]) < 1e-30f) q[i] = __fdividef(n, mu[i]);
  }
}

// The terms t = mu - n + n ln(n / mu) of N points in a bin with data, from
// d = n - mu, s = n + mu and q = n / mu: the atanh series where |d| < 0.1 s,
// else the direct form, with the quotient floored at 1e-30 (mu = 0 gives +inf).
// All lanes call this together (the bin, and so n, is the warp's); a form that
// none of the warp's points needs is not evaluated, nor (QUOT = false) is q
// formed for the series.  mu < 0 is left to the caller; n is at least 1e-30.
template <int N, bool QUOT>
__device__ __forceinline__ Vf<N> deviance_warp(Vf<N> d, Vf<N> s, float n, const float* mu, float* q) {
  float dv[N], sv[N], t[N];
  d.to(dv);
  s.to(sv);
  // clearly far from the data (the exact rule is the quotient's, below)
  bool far = true;
#pragma unroll
  for (int i = 0; i < N; ++i) far = far && fabsf(dv[i]) > 0.1001f * sv[i];
  bool near[N], all_near = false;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    near[i] = false;
    t[i] = 0.f;
  }
  if (!__all_sync(0xffffffffu, far)) {
    float vv[N];
#pragma unroll
    for (int i = 0; i < N; ++i) vv[i] = quotient(dv[i], sv[i]);
    const Vf<N> v = Vf<N>::of(vv), v2 = vmul(v, v);
    Vf<N> p = vfma(v2, Vf<N>::dup(1.f / 9.f), Vf<N>::dup(1.f / 7.f));
    p = vfma(v2, p, Vf<N>::dup(1.f / 5.f));
    p = vfma(v2, p, Vf<N>::dup(1.f / 3.f));
    vfma(d, v, vmul(vmul(vmul(Vf<N>::dup(2.f * n), v), v2), p)).to(t);
    all_near = true;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      near[i] = fabsf(vv[i]) < 0.1f;
      all_near = all_near && near[i];
    }
  }
  if (QUOT) quotients<N>(n, mu, q);
  if (!__all_sync(0xffffffffu, all_near)) {
    if (!QUOT) quotients<N>(n, mu, q);
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const float tl = __fmaf_rn(n, logf(fmaxf(q[i], 1e-30f)), -dv[i]);
      t[i] = near[i] ? t[i] : tl;
    }
  }
  return Vf<N>::of(t);
}

// The same terms for K bins of two points each without a branch per bin (few
// warps: the K x 2 terms' latencies overlap instead), the direct form skipped
// only if no term of the warp needs it; n[k] = 0 gives t = mu.
template <int K>
__device__ __forceinline__ void deviance_bins(const Vf<2>* d, const Vf<2>* s, const float* n, const float (*mu)[2],
                                              float (*q)[2], float (*t)[2]) {
  bool fine = true;
#pragma unroll
  for (int k = 0; k < K; ++k) fine = fine && !(fabsf(mu[k][0]) < 1e-30f) && !(fabsf(mu[k][1]) < 1e-30f);
  const bool scaled = !__all_sync(0xffffffffu, fine);
  bool near[K][2], all_near = true;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    float dv[2], sv[2], vv[2];
    d[k].to(dv);
    s[k].to(sv);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      vv[i] = quotient(dv[i], sv[i]);
      q[k][i] = quotient(n[k], mu[k][i]);
    }
    const Vf<2> v = Vf<2>::of(vv), v2 = vmul(v, v);
    Vf<2> p = vfma(v2, Vf<2>::dup(1.f / 9.f), Vf<2>::dup(1.f / 7.f));
    p = vfma(v2, p, Vf<2>::dup(1.f / 5.f));
    p = vfma(v2, p, Vf<2>::dup(1.f / 3.f));
    vfma(d[k], v, vmul(vmul(vmul(Vf<2>::dup(2.f * n[k]), v), v2), p)).to(t[k]);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      near[k][i] = fabsf(vv[i]) < 0.1f;
      all_near = all_near && (near[k][i] || n[k] == 0.f);
    }
  }
  if (scaled)
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
      for (int i = 0; i < 2; ++i)
        if (fabsf(mu[k][i]) < 1e-30f) q[k][i] = __fdividef(n[k], mu[k][i]);
  if (!__all_sync(0xffffffffu, all_near))
#pragma unroll
    for (int k = 0; k < K; ++k) {
      float dv[2];
      d[k].to(dv);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float tl = __fmaf_rn(n[k], logf(fmaxf(q[k][i], 1e-30f)), -dv[i]);
        t[k][i] = near[k][i] ? t[k][i] : tl;
      }
    }
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int i = 0; i < 2; ++i) t[k][i] = n[k] == 0.f ? mu[k][i] : t[k][i];
}

// Constants of one bin in shared memory: M row, n - mu_ref - b, n + mu_ref + b,
// n, mask; for two points a lane the factors are stored twice, as the packed
// instructions take them.
template <int N>
struct BinConsts;
template <>
struct BinConsts<1> {
  float4 a, b, c;
  __device__ __forceinline__ void set(const float4* g) { a = g[0]; b = g[1]; c = g[2]; }
  __device__ __forceinline__ Vf<1> m(int k) const {
    return {k == 0 ? a.x : k == 1 ? a.y : k == 2 ? a.z : k == 3 ? a.w : k == 4 ? b.x : k == 5 ? b.y : b.z};
  }
  __device__ __forceinline__ Vf<1> nb() const { return {b.w}; }
};
template <>
struct BinConsts<2> {
  ulonglong2 a, b, d, e;
  float4 c;
  __device__ __forceinline__ void set(const float4* g) {
    const float4 x = g[0], y = g[1];
    a = make_ulonglong2(pk(x.x, x.x), pk(x.y, x.y));
    b = make_ulonglong2(pk(x.z, x.z), pk(x.w, x.w));
    d = make_ulonglong2(pk(y.x, y.x), pk(y.y, y.y));
    e = make_ulonglong2(pk(y.z, y.z), pk(y.w, y.w));
    c = g[2];
  }
  __device__ __forceinline__ Vf<2> m(int k) const {
    return {k == 0 ? a.x : k == 1 ? a.y : k == 2 ? b.x : k == 3 ? b.y : k == 4 ? d.x : k == 5 ? d.y : e.x};
  }
  __device__ __forceinline__ Vf<2> nb() const { return {e.y}; }
};

// Dot product of a bin's M row with the points' seven coefficient deviations.
template <int N>
__device__ __forceinline__ Vf<N> row_dot(const BinConsts<N>& q, const Vf<N>* c) {
  Vf<N> dl = vmul(q.m(0), c[0]);
#pragma unroll
  for (int k = 1; k < kNB - 1; ++k) dl = vfma(q.m(k), c[k], dl);
  return dl;
}

// The same from the undoubled constants of a bin.
__device__ __forceinline__ Vf<2> row_dot(const float4& a, const float4& b, const Vf<2>* c) {
  Vf<2> dl = vmul(Vf<2>::dup(a.x), c[0]);
  dl = vfma(Vf<2>::dup(a.y), c[1], dl);
  dl = vfma(Vf<2>::dup(a.z), c[2], dl);
  dl = vfma(Vf<2>::dup(a.w), c[3], dl);
  dl = vfma(Vf<2>::dup(b.x), c[4], dl);
  dl = vfma(Vf<2>::dup(b.y), c[5], dl);
  return vfma(Vf<2>::dup(b.z), c[6], dl);
}

// The seven deviations (the constant monomial's is zero) of N points.
template <int N>
__device__ __forceinline__ void point_deviations(const float* theta, const int* p, int P, dfloat sin2w,
                                                 const CoefRef& cref, Vf<N>* c, Couplings* g) {
  float cc[N][kNB];
#pragma unroll
  for (int i = 0; i < N; ++i) {
#pragma unroll
    for (int b = 0; b < kNB; ++b) cc[i][b] = 0.f;
    g[i] = Couplings{0.f, 0.f, 0.f, 0.f, 0.f};
    if (p[i] < P) deviations(theta + (size_t)p[i] * 5, sin2w, cref, cc[i], g[i]);
  }
#pragma unroll
  for (int b = 0; b < kNB - 1; ++b) {
    float x[N];
#pragma unroll
    for (int i = 0; i < N; ++i) x[i] = cc[i][b < 6 ? b : 7];
    c[b] = Vf<N>::of(x);
  }
}

// The value and gradient of one point from the sums of its four residues.
struct LinSums {
  dfloat acc[4];
  bool infinite;
  float gb[4][kNB - 1];
};
template <bool GRAD>
__device__ __forceinline__ void finish_point(const LinSums& r, const Couplings& g, const double* c_data, double* out,
                                             double* grad, unsigned* status) {
  const dfloat a = df_add(df_add(r.acc[0], r.acc[1]), df_add(r.acc[2], r.acc[3]));
  if (r.infinite) atomicOr(status, kStatusDomain);
  *out = r.infinite ? __longlong_as_double(0x7ff0000000000000LL) : 2.0 * ((double)a.hi + (double)a.lo) + *c_data;
  if (GRAD) {
    float b[kNB - 1];
#pragma unroll
    for (int k = 0; k < kNB - 1; ++k) b[k] = (r.gb[0][k] + r.gb[1][k]) + (r.gb[2][k] + r.gb[3][k]);
    grad[0] = 2.0 * (2.0 * (double)g.gle * b[0] - (double)g.gre * b[2]);
    grad[1] = 2.0 * (2.0 * (double)g.gre * b[1] - (double)g.gle * b[2]);
    grad[2] = 2.0 * (2.0 * (double)g.glt * b[3] - (double)g.grt * b[5]);
    grad[3] = 2.0 * (2.0 * (double)g.grt * b[4] - (double)g.glt * b[5]);
    grad[4] = 2.0 * (2.0 * (double)g.mu * b[6]);
  }
}

// Batches that fill the GPU at a warp per residue: warp w of a block takes bins
// w, w + 4, ... of 32 N points.  N = 2 from 128 points an SM on (seven blocks
// share an SM; 65,536 points with gradient on the solar set: 253 us, N = 1
// 289 us); below that the second point's warps are missed more than its
// packed instructions help (see launch_linear).
template <bool GRAD, int N>
__global__ void __launch_bounds__(kLinThreads, N == 2 ? 7 : 8)
linear_loglik_kernel(const float* __restrict__ theta, int P, dfloat sin2w, CoefRef cref,
                     const float4* __restrict__ consts, int n_rec, const double* __restrict__ c_data,
                     double* __restrict__ out, double* __restrict__ grad, unsigned* __restrict__ status) {
  __shared__ BinConsts<N> sc[kLinChunk];
  __shared__ float2 sacc[4][N][32];
  __shared__ int sinf_[4][N][32];
  __shared__ float sgb[GRAD ? 4 : 1][kNB - 1][N][32];
  const int quarter = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int p[N];
#pragma unroll
  for (int i = 0; i < N; ++i) p[i] = blockIdx.x * (32 * N) + 32 * i + lane;
  Vf<N> c[kNB - 1], gb[kNB - 1];
  Couplings g[N];
  point_deviations<N>(theta, p, P, sin2w, cref, c, g);
#pragma unroll
  for (int b = 0; b < kNB - 1; ++b) gb[b] = Vf<N>::dup(0.f);
  dfloat acc[N];
  bool infinite[N];
  float mneg[N];  // smallest mu of the active bins (below 0: outside the domain)
#pragma unroll
  for (int i = 0; i < N; ++i) {
    acc[i] = {0.f, 0.f};
    infinite[i] = false;
    mneg[i] = 0.f;
  }
  for (int j0 = 0; j0 < n_rec; j0 += kLinChunk) {
    const int cnt = min(kLinChunk, n_rec - j0);
    __syncthreads();
    for (int k = threadIdx.x; k < cnt; k += kLinThreads) sc[k].set(consts + 3 * (size_t)(j0 + k));
    __syncthreads();
    for (int j1 = quarter; j1 < cnt; j1 += 64) {  // FP32 sums over 16 bins, added up in double-float
      Vf<N> ts = Vf<N>::dup(0.f);
#pragma unroll (N == 2 ? 2 : 4)
      for (int j = j1; j < min(cnt, j1 + 64); j += 4) {
        const BinConsts<N>& q = sc[j];
        if (q.c.z == 0.f) continue;  // masked
        const Vf<N> dl = row_dot<N>(q, c);
        const float n = q.c.y;
        const Vf<N> d = vsub(q.nb(), dl), mu = vsub(Vf<N>::dup(n), d);
        float m[N], r[N];
        mu.to(m);
        if (n == 0.f) {  // no data: t = mu, and 1 - n / mu is 1 (NaN at mu = 0)
          ts = vadd(ts, mu);
          if (GRAD)
#pragma unroll
            for (int i = 0; i < N; ++i) r[i] = m[i] == 0.f || m[i] != m[i] ? __int_as_float(0x7fc00000) : 1.f;
        } else {
          float nq[N];
          ts = vadd(ts, deviance_warp<N, GRAD>(d, vadd(Vf<N>::dup(q.c.x), dl), n, m, nq));
          if (GRAD)
#pragma unroll
            for (int i = 0; i < N; ++i) r[i] = __fsub_rn(1.f, nq[i]);
        }
#pragma unroll
        for (int i = 0; i < N; ++i) mneg[i] = fminf(mneg[i], m[i]);
        if (GRAD) {
          const Vf<N> rr = Vf<N>::of(r);
#pragma unroll
          for (int b = 0; b < kNB - 1; ++b) gb[b] = vfma(q.m(b), rr, gb[b]);
        }
      }
      float t[N];
      ts.to(t);
#pragma unroll
      for (int i = 0; i < N; ++i) {
        if (isinf(t[i])) infinite[i] = true;
        else acc[i] = df_add(acc[i], t[i]);
      }
    }
  }
  // combine the four warps' sums of each point
#pragma unroll
  for (int i = 0; i < N; ++i) {
    sacc[quarter][i][lane] = make_float2(acc[i].hi, acc[i].lo);
    sinf_[quarter][i][lane] = infinite[i] || mneg[i] < 0.f;
  }
  if (GRAD)
#pragma unroll
    for (int b = 0; b < kNB - 1; ++b) {
      float x[N];
      gb[b].to(x);
#pragma unroll
      for (int i = 0; i < N; ++i) sgb[quarter][b][i][lane] = x[i];
    }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < N; ++i) {
    if (quarter != i || p[i] >= P) continue;  // warp i finishes point group i
    LinSums r;
    r.infinite = false;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      r.acc[w] = dfloat{sacc[w][i][lane].x, sacc[w][i][lane].y};
      r.infinite = r.infinite || sinf_[w][i][lane] != 0;
      if (GRAD)
#pragma unroll
        for (int k = 0; k < kNB - 1; ++k) r.gb[w][k] = sgb[w][k][i][lane];
    }
    finish_point<GRAD>(r, g[i], c_data, out + p[i], GRAD ? grad + (size_t)p[i] * 5 : nullptr, status);
  }
}

// Small batches: 2 L points a block.  The terms of a round of 64 bins are
// formed by all 512 threads (L lanes of two points, L / 8 bins each), left in
// shared memory, and added up in the same order as above by a thread per
// (point, residue, share of the chains).  A block's time is its instructions,
// so few points go to many SMs (500 points with gradient on the solar set:
// 85 us at four lanes a point, 80 us at L = 32, 29 us at L = 8).
template <int L>
struct SplitMap {
  static constexpr int kPoints = 2 * L, kBins = L / 8;
  int pt, q, i0;      // terms: points pt and L + pt, bins q + 4 (i0 + u) of a round
  int cpt, cq, ck;    // chains: point, residue, share
  bool chain;
  __device__ __forceinline__ SplitMap() {
    const int lane = threadIdx.x & 31, slot = (threadIdx.x >> 5) * (32 / L) + lane / L;
    pt = lane % L;
    q = slot & 3;
    i0 = (slot >> 2) * kBins;
    cpt = threadIdx.x % kPoints;
    cq = (threadIdx.x / kPoints) & 3;
    ck = threadIdx.x / (4 * kPoints);
    chain = ck < 2;
  }
  __device__ __forceinline__ int bin(int r, int u) const { return r * kSplitRound + q + 4 * (i0 + u); }
};
// Term (round parity, kind, residue, i, point) of bin q + 4 i of a round.
template <int L>
__device__ __forceinline__ float* split_term(float* terms, int par, int k, int q, int i) {
  return terms + ((((par * 2 + k) * 4 + q) * 16 + i) * (2 * L));
}

template <bool GRAD, int L>
__global__ void __launch_bounds__(kSplitThreads, L == 16 ? 2 : 1)
linear_split_kernel(const float* __restrict__ theta, int P, dfloat sin2w, CoefRef cref,
                    const float4* __restrict__ consts, int n_rec, const double* __restrict__ c_data,
                    double* __restrict__ out, double* __restrict__ grad, unsigned* __restrict__ status) {
  constexpr int PB = SplitMap<L>::kPoints, K = SplitMap<L>::kBins;
  extern __shared__ float4 sc[];  // [min(n_rec, kSplitChunk)][3], then the terms of two rounds
  __shared__ float2 sacc[4][PB];
  __shared__ int sinf_[4][PB];
  __shared__ float sgb[GRAD ? 4 : 1][kNB - 1][PB];
  float* terms = reinterpret_cast<float*>(sc + 3 * (size_t)min(n_rec, kSplitChunk));
  const SplitMap<L> S;
  const int p0 = blockIdx.x * PB, p[2] = {p0 + S.pt, p0 + L + S.pt};
  Vf<2> c[kNB - 1];
  {
    Couplings g[2];
    point_deviations<2>(theta, p, P, sin2w, cref, c, g);
  }
  dfloat acc = {0.f, 0.f};
  bool infinite = false;
  float gb[4] = {0.f, 0.f, 0.f, 0.f};
  for (int j0 = 0; j0 < n_rec; j0 += kSplitChunk) {
    const int cnt = min(kSplitChunk, n_rec - j0);
    __syncthreads();
    for (int k = threadIdx.x; k < 3 * cnt; k += kSplitThreads) sc[k] = consts[3 * (size_t)j0 + k];
    __syncthreads();
    const int rounds = (cnt + kSplitRound - 1) / kSplitRound;
    for (int r = 0; r <= rounds; ++r) {
      if (r < rounds) {
        Vf<2> d[K], sm[K];
        float n[K], mu[K][2], q[K][2], t[K][2];
        bool on[K];
#pragma unroll
        for (int u = 0; u < K; ++u) {
          const int j = S.bin(r, u), jc = min(j, cnt - 1);
          const float4 a = sc[3 * jc], b = sc[3 * jc + 1], e = sc[3 * jc + 2];
          const Vf<2> dl = row_dot(a, b, c);
          n[u] = e.y;
          on[u] = j < cnt && e.z != 0.f;
          d[u] = vsub(Vf<2>::dup(b.w), dl);
          sm[u] = vadd(Vf<2>::dup(e.x), dl);
          vsub(Vf<2>::dup(e.y), d[u]).to(mu[u]);
        }
        deviance_bins<K>(d, sm, n, mu, q, t);
#pragma unroll
        for (int u = 0; u < K; ++u) {
          float *tv = split_term<L>(terms, r & 1, 0, S.q, S.i0 + u) + S.pt;
          float *tr = split_term<L>(terms, r & 1, 1, S.q, S.i0 + u) + S.pt;
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const float m = mu[u][k];
            tv[L * k] = !on[u] ? 0.f : m < 0.f ? __int_as_float(0x7f800000) : t[u][k];
            if (GRAD) {  // 1 - n / mu: 1 without data (NaN at mu = 0)
              const float x0 = m == 0.f || m != m ? __int_as_float(0x7fc00000) : 1.f;
              tr[L * k] = !on[u] ? 0.f : n[u] == 0.f ? x0 : __fsub_rn(1.f, q[u][k]);
            }
          }
        }
      }
      if (r > 0 && S.chain && (GRAD || S.ck == 0)) {
        // in order of the bins: the value and three of the gradient's sums, or its other four
        const float* tv = split_term<L>(terms, (r - 1) & 1, 0, S.cq, 0) + S.cpt;
        const float* tr = split_term<L>(terms, (r - 1) & 1, 1, S.cq, 0) + S.cpt;
        float ts = 0.f;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int j = min((r - 1) * kSplitRound + S.cq + 4 * i, cnt - 1);
          const float x = GRAD ? tr[i * PB] : 0.f;
          if (S.ck == 0) {
            ts = __fadd_rn(ts, tv[i * PB]);
            if (GRAD) {
              const float4 a = sc[3 * j];
              gb[0] = __fmaf_rn(a.x, x, gb[0]);
              gb[1] = __fmaf_rn(a.y, x, gb[1]);
              gb[2] = __fmaf_rn(a.z, x, gb[2]);
            }
          } else {
            const float4 b = sc[3 * j + 1];
            gb[0] = __fmaf_rn(sc[3 * j].w, x, gb[0]);
            gb[1] = __fmaf_rn(b.x, x, gb[1]);
            gb[2] = __fmaf_rn(b.y, x, gb[2]);
            gb[3] = __fmaf_rn(b.z, x, gb[3]);
          }
        }
        if (S.ck == 0) {
          if (isinf(ts)) infinite = true;
          else acc = df_add(acc, ts);
        }
      }
      __syncthreads();
    }
  }
  if (S.ck == 0) {
    sacc[S.cq][S.cpt] = make_float2(acc.hi, acc.lo);
    sinf_[S.cq][S.cpt] = infinite;
  }
  if (GRAD && S.chain)
#pragma unroll
    for (int b = 0; b < 4; ++b)
      if (S.ck == 1 || b < 3) sgb[S.cq][S.ck * 3 + b][S.cpt] = gb[b];
  __syncthreads();
  const int q = threadIdx.x;
  if (q >= PB || p0 + q >= P) return;
  LinSums r;
  r.infinite = false;
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    r.acc[w] = dfloat{sacc[w][q].x, sacc[w][q].y};
    r.infinite = r.infinite || sinf_[w][q] != 0;
    if (GRAD)
#pragma unroll
      for (int k = 0; k < kNB - 1; ++k) r.gb[w][k] = sgb[w][k][q];
  }
  float cc[kNB];
  Couplings g;
  deviations(theta + (size_t)(p0 + q) * 5, sin2w, cref, cc, g);
  finish_point<GRAD>(r, g, c_data, out + p0 + q, GRAD ? grad + (size_t)(p0 + q) * 5 : nullptr, status);
}

constexpr int kNewton = 8;  // Newton steps for the normalisation (quadratic convergence from alpha = 1)

// Profiled evaluation: min over alpha >= 0 of -2 ln L(alpha mu_sig + b) plus
// ((alpha - 1)/sigma)^2 when sigma > 0, with mu_sig = mu_ref + M (c - c_ref).
// Newton on the convex objective, g = 2 sum s (1 - n/mu) + 2 (alpha - 1)/sigma^2,
// h = 2 sum n s^2 / mu^2 + 2 / sigma^2, each step one pass over the bins
// (mu_sig recomputed from the coefficients); then the deviance at alpha.  A
// step that changes no point of the block ends the iteration: every further
// one would give the same alpha.
//
// The sums of g and h run over the bins of one residue modulo 4 in order, in
// FP32: a chain per point that a grid of few points cannot fill the GPU with
// (8191 points at a warp per chain: 1.7 warps a scheduler, 900 us).  So the
// terms are formed and added as in linear_split_kernel, a thread per (point,
// residue, g or h) adding a round's sixteen terms in order while the next
// round's are formed.  The last pass sums its deviances the same way.
template <int L>
__global__ void __launch_bounds__(kSplitThreads, 1)
linear_profiled_kernel(const float* __restrict__ theta, int P, dfloat sin2w, CoefRef cref,
                       const float4* __restrict__ consts, const float4* __restrict__ constp, int n_rec,
                       float inv_var, const double* __restrict__ c_data, double* __restrict__ out,
                       double* __restrict__ alpha_out, unsigned* __restrict__ status) {
  constexpr int PB = SplitMap<L>::kPoints, K = SplitMap<L>::kBins;
  extern __shared__ float4 sc[];  // [min(n_rec, kProfChunk)][3], then the terms of two rounds
  __shared__ float sums[4][2][PB];
  __shared__ float salpha[PB];
  __shared__ float2 sacc[4][PB];
  __shared__ int sinf_[4][PB];
  float* terms = reinterpret_cast<float*>(sc + 3 * (size_t)min(n_rec, kProfChunk));
  const SplitMap<L> S;
  const int p0 = blockIdx.x * PB, p[2] = {p0 + S.pt, p0 + L + S.pt};
  Vf<2> c[kNB - 1];
  {
    Couplings g[2];
    point_deviations<2>(theta, p, P, sin2w, cref, c, g);
  }
  const bool resident = n_rec <= kProfChunk;
  auto stage = [&](int j0, int cnt, bool first) {
    if (resident && !first) return;
    __syncthreads();
    for (int k = threadIdx.x; k < cnt; k += kSplitThreads) {
      sc[3 * k] = consts[3 * (size_t)(j0 + k)];
      sc[3 * k + 1] = consts[3 * (size_t)(j0 + k) + 1];
      sc[3 * k + 2] = constp[j0 + k];
    }
    __syncthreads();
  };
  auto signal = [&](int j) {  // mu_sig of the lane's two points
    return vadd(Vf<2>::dup(sc[3 * j + 2].x), row_dot(sc[3 * j], sc[3 * j + 1], c));
  };
  float alpha[2] = {1.f, 1.f};
  for (int it = 0; it < kNewton; ++it) {
    float sum = 0.f;  // this thread's chain
    const Vf<2> al = Vf<2>::of(alpha);
    for (int j0 = 0; j0 < n_rec; j0 += kProfChunk) {
      const int cnt = min(kProfChunk, n_rec - j0);
      stage(j0, cnt, it == 0);
      const int rounds = (cnt + kSplitRound - 1) / kSplitRound;
      for (int r = 0; r <= rounds; ++r) {
        if (r < rounds) {
          float sv[K][2], mu[K][2], x[K][2], n[K];
          bool on[K], fine = true;
#pragma unroll
          for (int u = 0; u < K; ++u) {
            const int j = S.bin(r, u), jc = min(j, cnt - 1);
            const float4 q = sc[3 * jc + 2];
            const Vf<2> s = signal(jc);
            s.to(sv[u]);
            vfma(al, s, Vf<2>::dup(q.y)).to(mu[u]);
            n[u] = q.z;
            on[u] = j < cnt && q.z >= 0.f;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              x[u][k] = quotient(q.z, mu[u][k]);  // n / mu
              fine = fine && !(fabsf(mu[u][k]) < 1e-30f);
            }
          }
          if (!__all_sync(0xffffffffu, fine))
#pragma unroll
            for (int u = 0; u < K; ++u)
#pragma unroll
              for (int k = 0; k < 2; ++k)
                if (fabsf(mu[u][k]) < 1e-30f) x[u][k] = __fdividef(n[u], mu[u][k]);
#pragma unroll
          for (int u = 0; u < K; ++u) {
            float *a = split_term<L>(terms, r & 1, 0, S.q, S.i0 + u) + S.pt;
            float *b = split_term<L>(terms, r & 1, 1, S.q, S.i0 + u) + S.pt;
            float h[2] = {0.f, 0.f};
            if (n[u] > 0.f) {  // no quotient without data
#pragma unroll
              for (int k = 0; k < 2; ++k) {
                const bool live = mu[u][k] > 0.f;
                x[u][k] = live ? x[u][k] : 0.f;
                h[k] = live ? __fdiv_rn(__fmul_rn(__fmul_rn(x[u][k], sv[u][k]), sv[u][k]), mu[u][k]) : 0.f;
              }
            } else {
              x[u][0] = x[u][1] = 0.f;
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              a[L * k] = on[u] ? __fmul_rn(sv[u][k], __fsub_rn(1.f, x[u][k])) : 0.f;
              b[L * k] = on[u] ? h[k] : 0.f;
            }
          }
        }
        if (r > 0 && S.chain) {  // the previous round's terms, complete since the last barrier
          const float* t = split_term<L>(terms, (r - 1) & 1, S.ck, S.cq, 0) + S.cpt;
#pragma unroll
          for (int i = 0; i < 16; ++i) sum = __fadd_rn(sum, t[i * PB]);
        }
        __syncthreads();
      }
    }
    if (S.chain) sums[S.cq][S.ck][S.cpt] = sum;
    __syncthreads();
    bool same = true;
    if (threadIdx.x < PB) {
      const int q = threadIdx.x;
      const float a = it == 0 ? 1.f : salpha[q];
      const float G = (sums[0][0][q] + sums[1][0][q]) + (sums[2][0][q] + sums[3][0][q]);
      const float H = (sums[0][1][q] + sums[1][1][q]) + (sums[2][1][q] + sums[3][1][q]);
      const float gg = 2.f * G + 2.f * (a - 1.f) * inv_var, hh = 2.f * H + 2.f * inv_var;
      float next = hh > 0.f ? a - gg / hh : (gg > 0.f ? 0.f : a);
      next = fmaxf(next, 0.f);
      same = next == a;
      salpha[q] = next;
    }
    same = __syncthreads_and(same);
    alpha[0] = salpha[S.pt];
    alpha[1] = salpha[L + S.pt];
    if (same) break;
  }
  // deviance at alpha: FP32 sums over the sixteen bins of a residue in a round,
  // added up in double-float by the warps of the first chain kind
  dfloat acc = {0.f, 0.f};
  bool infinite = false;
  for (int j0 = 0; j0 < n_rec; j0 += kProfChunk) {
    const int cnt = min(kProfChunk, n_rec - j0);
    stage(j0, cnt, false);
    const int rounds = (cnt + kSplitRound - 1) / kSplitRound;
    for (int r = 0; r <= rounds; ++r) {
      if (r < rounds) {
        Vf<2> d[K], sm[K];
        float n[K], mu[K][2], m[K][2], q[K][2], t[K][2];
        bool on[K];
#pragma unroll
        for (int u = 0; u < K; ++u) {
          const int j = S.bin(r, u), jc = min(j, cnt - 1);
          const float4 e = sc[3 * jc + 2];
          on[u] = j < cnt && e.z >= 0.f;
          n[u] = fmaxf(e.z, 0.f);
          const Vf<2> mv = vfma(Vf<2>::of(alpha), signal(jc), Vf<2>::dup(e.y)), n2 = Vf<2>::dup(n[u]);
          mv.to(mu[u]);
          d[u] = vsub(n2, mv);
          sm[u] = vadd(n2, mv);
          vsub(n2, d[u]).to(m[u]);
        }
        deviance_bins<K>(d, sm, n, m, q, t);
#pragma unroll
        for (int u = 0; u < K; ++u) {
          float* a = split_term<L>(terms, r & 1, 0, S.q, S.i0 + u) + S.pt;
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const float x = n[u] == 0.f ? mu[u][k] : m[u][k];
            const bool out_of = x < 0.f || (x == 0.f && n[u] > 0.f);
            a[L * k] = !on[u] ? 0.f : out_of ? __int_as_float(0x7f800000) : t[u][k];
          }
        }
      }
      if (r > 0 && S.ck == 0) {
        const float* t = split_term<L>(terms, (r - 1) & 1, 0, S.cq, 0) + S.cpt;
        float ts = 0.f;
#pragma unroll
        for (int i = 0; i < 16; ++i) ts = __fadd_rn(ts, t[i * PB]);
        if (isinf(ts)) infinite = true;
        else acc = df_add(acc, ts);
      }
      __syncthreads();
    }
  }
  if (S.ck == 0) {
    sacc[S.cq][S.cpt] = make_float2(acc.hi, acc.lo);
    sinf_[S.cq][S.cpt] = infinite;
  }
  __syncthreads();
  const int q = threadIdx.x, pq = blockIdx.x * PB + q;
  if (q >= PB || pq >= P) return;
  auto ap = [&](int w) { return dfloat{sacc[w][q].x, sacc[w][q].y}; };
  acc = df_add(df_add(ap(0), ap(1)), df_add(ap(2), ap(3)));
  infinite = (sinf_[0][q] | sinf_[1][q] | sinf_[2][q] | sinf_[3][q]) != 0;
  const double a = (double)salpha[q];
  const double pull = (double)inv_var * (a - 1.0) * (a - 1.0);
  const double v = infinite ? __longlong_as_double(0x7ff0000000000000LL)
                            : 2.0 * ((double)acc.hi + (double)acc.lo) + *c_data + pull;
  if (infinite) atomicOr(status, kStatusDomain);
  out[pq] = v;
  if (alpha_out) alpha_out[pq] = a;
}

// Dynamic shared memory of the split kernels: the constants of up to `chunk` bins and the terms of two rounds.
template <int L>
constexpr size_t split_smem(int n_rec, int chunk) {
  return 3 * sizeof(float4) * (size_t)(n_rec < chunk ? n_rec : chunk) +
         sizeof(float) * 2 * 2 * kSplitRound * SplitMap<L>::kPoints;
}

template <bool GRAD, int L>
void launch_split(const srw_ctx* h, const float* theta, int P, double* out, double* grad, cudaStream_t s) {
  constexpr int PB = SplitMap<L>::kPoints;
  linear_split_kernel<GRAD, L><<<(P + PB - 1) / PB, kSplitThreads, split_smem<L>(h->n_rec, kSplitChunk), s>>>(
      theta, P, df_from_double(h->sin2w), h->cref, h->d_lin, h->n_rec, h->d_cdata, out, grad, h->d_status);
}

template <bool GRAD, int N>
void launch_warps(const srw_ctx* h, const float* theta, int P, double* out, double* grad, cudaStream_t s) {
  linear_loglik_kernel<GRAD, N><<<(P + 32 * N - 1) / (32 * N), kLinThreads, 0, s>>>(
      theta, P, df_from_double(h->sin2w), h->cref, h->d_lin, h->n_rec, h->d_cdata, out, grad, h->d_status);
}

template <bool GRAD>
void launch_linear(const srw_ctx* h, const float* theta, int P, double* out, double* grad, cudaStream_t s) {
  // The lines lie where the one side becomes the faster; the first two are also
  // whole waves, one block of 16 points an SM (L = 8), then two of 32 (L = 16).
  // us on 2048 bins, value only / with gradient, back to back:
  //   points      L = 8      L = 16   one a lane   two a lane
  //    2432     21 / 29     31 / 48     88 / 95     91 / 117
  //    9727     54 / 107    48 / 75     91 / 98     92 / 118
  //   12,000    66 / 132    71 / 111    93 / 103    98 / 128
  //   19,000   101 / 208    91 / 144    99 / 111    99 / 129
  //   40,000   207 / 437   195 / 311   194 / 220   140 / 189
  // (Values alone from 2433 to about 7000 points would be 2 to 4 us faster at L = 8.)
  if (P <= 16 * h->sm_count) launch_split<GRAD, 8>(h, theta, P, out, grad, s);
  else if (P < (GRAD ? 64 : 128) * h->sm_count) launch_split<GRAD, 16>(h, theta, P, out, grad, s);
  else if (GRAD && P < 128 * h->sm_count) launch_warps<true, 1>(h, theta, P, out, grad, s);
  else launch_warps<GRAD, 2>(h, theta, P, out, grad, s);
}

template <int L>
void launch_profiled(const srw_ctx* h, const float* theta, int P, float inv_var, double* out, double* alpha,
                     cudaStream_t s) {
  constexpr int PB = SplitMap<L>::kPoints;
  linear_profiled_kernel<L><<<(P + PB - 1) / PB, kSplitThreads, split_smem<L>(h->n_rec, kProfChunk), s>>>(
      theta, P, df_from_double(h->sin2w), h->cref, h->d_lin, h->d_linp, h->n_rec, inv_var, h->d_cdata, out, alpha,
      h->d_status);
}

template <class F>
cudaError_t allow_smem(F* f, size_t bytes) {
  return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace

cudaError_t launch_linear_profiled(const srw_ctx* h, const float* theta, int P, double sigma_alpha, double* out,
                                   double* alpha, cudaStream_t s) {
  const float inv_var = sigma_alpha > 0.0 ? (float)(1.0 / (sigma_alpha * sigma_alpha)) : 0.f;
  // the fewest points a block that still gives every SM at most one
  if (P <= 16 * h->sm_count) launch_profiled<8>(h, theta, P, inv_var, out, alpha, s);
  else if (P <= 32 * h->sm_count) launch_profiled<16>(h, theta, P, inv_var, out, alpha, s);
  else launch_profiled<32>(h, theta, P, inv_var, out, alpha, s);
  return launch_result();
}

cudaError_t launch_linear_m(srw_ctx* h, cudaStream_t s) {
  cudaError_t e = allow_smem(linear_profiled_kernel<8>, split_smem<8>(kProfChunk, kProfChunk));
  if (e == cudaSuccess) e = allow_smem(linear_profiled_kernel<16>, split_smem<16>(kProfChunk, kProfChunk));
  if (e == cudaSuccess) e = allow_smem(linear_profiled_kernel<32>, split_smem<32>(kProfChunk, kProfChunk));
  if (e == cudaSuccess) e = allow_smem(linear_split_kernel<true, 8>, split_smem<8>(kSplitChunk, kSplitChunk));
  if (e == cudaSuccess) e = allow_smem(linear_split_kernel<false, 8>, split_smem<8>(kSplitChunk, kSplitChunk));
  if (e == cudaSuccess) e = allow_smem(linear_split_kernel<true, 16>, split_smem<16>(kSplitChunk, kSplitChunk));
  if (e == cudaSuccess) e = allow_smem(linear_split_kernel<false, 16>, split_smem<16>(kSplitChunk, kSplitChunk));
  if (e != cudaSuccess) return e;
  linear_m_kernel<<<h->n_rec, 256, 0, s>>>(h->d_R, h->ld_r, h->n_t, h->d_basis, h->d_ssm64, h->d_esm64, h->d_linM);
  return launch_result();
}

cudaError_t launch_linear_consts(srw_ctx* h, cudaStream_t s) {
  linear_consts_kernel<<<(h->n_rec + 255) / 256, 256, 0, s>>>(h->d_linM, h->d_n64, h->d_bref64, h->d_muref64, h->d_mask,
                                                             h->n_rec, h->d_lin, h->d_linp);
  return launch_result();
}

cudaError_t launch_linear_loglik(const srw_ctx* h, const float* theta, int P, double* out, double* grad,
                                 cudaStream_t s) {
  if (grad) launch_linear<true>(h, theta, P, out, grad, s);
  else launch_linear<false>(h, theta, P, out, nullptr, s);
  return launch_result();
}

}  // namespace srw
