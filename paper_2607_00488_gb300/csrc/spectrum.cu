// Recoil-spectrum kernels.
//
// The recoil spectrum of one true-recoil bin i is (Sec. III.A, eq. fT, with
// the cross sections of Sec. II, eqs. sm_cross_section, g_tilde, xs_mm,
// xs_total), in units of sigma0 = 2 G_F^2 m_e / pi:
//
//   S_i = sum_nodes w_n sum_alpha P_alpha(E_n) int_a^b dT [ gL_a^2
//           + gR_a^2 (1 - T/E)^2 - gL_a gR_a m_e T / E^2 ]
//       + kappa mu_hat^2 sum_nodes w_n int_a^b dT (1/T - 1/E)
//
// with a = max(T_lo, t_min), b = min(T_hi, T_max(E_n)) and
// T_max(E) = 2 E^2 / (m_e + 2E).  The integrals are closed forms:
//   int 1            = b - a                       (I0)
//   int T            = (b - a)(a + b) / 2          (I1)
//   int (1 - T/E)^2  = (b - a)(u^2 + u v + v^2)/3, u = 1 - a/E, v = 1 - b/E
//   int (1/T - 1/E)  = log(b/a) - (b - a)/E
// (the (1 - T/E)^2 form avoids the cancellation of expanding the cube).
//
// Nodes are sorted by T_max descending, so the nodes that can reach bin i
// are a prefix [0, bin_count[i]).

#include "dfloat.cuh"
#include "srw_internal.h"

namespace srw {
namespace {

constexpr int kBasisThreads = 256;

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---------------------------------------------------------------------------
// G0: FP64 coefficient spectra B[8][n_t] (create time, theta independent).
// One block per recoil bin; threads stride over the contributing nodes;
// fixed-order block reduction (deterministic).  FP64 throughout, including
// the near-threshold 1/T magnetic-moment integrals.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kBasisThreads)
basis_fp64_kernel(ModelView m, double gl_mu, double gr_mu, double kappa, double* __restrict__ basis) {
  const int i = blockIdx.x;
  const int n_nodes = m.n_nodes;
  const double lo = m.bin64[i], hi = m.bin64[m.n_t + i];
  const double t_min = m.t_min64;
  const int count = m.bin_count[i];
  double acc[kNB];
#pragma unroll
  for (int b = 0; b < kNB; ++b) acc[b] = 0.0;

  for (int n = threadIdx.x; n < count; n += blockDim.x) {
    const double e = m.node64[n];
    const double wpe = m.node64[n_nodes + n], wpm = m.node64[2 * n_nodes + n];
    const double wpt = m.node64[3 * n_nodes + n], w = m.node64[4 * n_nodes + n];
    const double tmax = 2.0 * e * e / (kMe + 2.0 * e);
    double i0, irr, ilr, imm;
    if (m.midpoint) {
      const double tc = 0.5 * (lo + hi);
      if (!(tc >= t_min && tc < tmax)) continue;
      const double dt = hi - lo, y = 1.0 - tc / e;
      i0 = dt;
      irr = dt * y * y;
      ilr = dt * kMe * tc / (e * e);
      imm = dt * (1.0 / tc - 1.0 / e);
    } else {
      const double a = fmax(lo, t_min), b = fmin(hi, tmax);
      if (!(b > a)) continue;
      const double d = b - a, u = 1.0 - a / e, v = 1.0 - b / e;
      i0 = d;
      irr = d * (u * u + u * v + v * v) / 3.0;
      ilr = kMe * d * (a + b) / (2.0 * e * e);
      imm = log1p(d / a) - d / e;
    }
    acc[0] += wpe * i0;
    acc[1] += wpe * irr;
    acc[2] += wpe * ilr;
    acc[3] += wpt * i0;
    acc[4] += wpt * irr;
    acc[5] += wpt * ilr;
    acc[6] += wpm * (gl_mu * gl_mu * i0 + gr_mu * gr_mu * irr - gl_mu * gr_mu * ilr);
    acc[7] += w * kappa * imm;
  }

  __shared__ double red[kBasisThreads / 32][kNB];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int b = 0; b < kNB; ++b) {
    const double v = warp_sum_d(acc[b]);
    if (lane == 0) red[warp][b] = v;
  }
  __syncthreads();
  if (threadIdx.x < kNB) {
    double s = 0.0;
    for (int w = 0; w < kBasisThreads / 32; ++w) s += red[w][threadIdx.x];
    basis[threadIdx.x * m.n_t + i] = s;
  }
}

// ---------------------------------------------------------------------------
// G1: single-point spectrum + weights (the per-theta "physics update"), from
// the cross-section integrals of every node at this theta.
//
// Nodes are sorted by T_max, so the nodes that cover bin i whole are a prefix
// [0, full_i), and over a whole bin the integrals are polynomials in the bin's
// edges whose coefficients depend on the node alone.  With r = 1/E and the
// node's coupling-weighted a0 = sum w P gL^2, a1 = sum w P gR^2,
// a2 = sum w P gL gR and a3 = w kappa mu^2,
//   S_i = I0_i [X - p_i Y + q_i Z] + L_i V + sum of the clipped nodes,
//   X = sum (a0 + a1 - a3 r), Y = sum r (a1 + a2 m_e r / 2), Z = sum a1 r^2, V = sum a3
// over the prefix, with {I0, p, q, L} = {b - a, a + b, (a^2 + a b + b^2) / 3,
// log(b / a)} of the bin (midpoint mode: {dt, 2 tc, tc^2, dt / tc}).  So one
// scan over the nodes serves every bin: n_nodes + n_t terms instead of
// n_nodes x n_t.  Expanding (1 - T/E)^2 cancels to about
// (m_e / (m_e + 2E))^2 of its terms (2e-4 at the hep endpoint), which is why
// the sums are FP64; the nodes that end inside bin i, [full_i, count_i), are
// summed apart (a scan that starts again with every bin, in tiles of 32), so
// that a bin without nodes stays an exact zero.
//
// Two kernels, the second and the fold behind it launched programmatically.
// moments_kernel: one block of two warps per chunk of nodes writes the prefix
// sums inside its chunk and the chunk's totals (at most kMaxChunks, chunks of 32
// nodes up to 8192 nodes).  bins_kernel: every block scans the totals again, one
// warp per quantity, and evaluates kBinsPerBlock bins.  Both are bound by the
// chain of FP64 instructions of a warp (64 cycles each on an SM sub-partition,
// dependent or not, measured), so the work is spread thin: small chunks and
// blocks, the quantities of a chunk over two warps.
//
// Solar set (8003 nodes), device time per call of back-to-back calls, against a
// kernel over all (node, bin) pairs in FP32 (clusters of four blocks per eight
// bins): S at 4096 bins 34.8 -> 10.3 us, expected counts 49.2 -> 20.4 us; S at
// 257 bins 10.2 -> 10.3 us.  Letting bins_kernel start at the top of
// moments_kernel instead of at its end gave 20.5 us (S at 4096 bins), an
// ordinary launch 12.4 us.  A line (1 node, 256 bins) takes the one-kernel form,
// 7.5 -> 7.4 us, expected counts 13.0 -> 9.6 us; with the two kernels S took
// 10.2 us.
// ---------------------------------------------------------------------------
constexpr int kMaxChunks = kSpecChunks;
constexpr int kBinsPerBlock = 16;
constexpr int kLanesPerBin = 8;  // clipped nodes of a bin
constexpr int kBinThreads = kBinsPerBlock * kLanesPerBin;
static_assert(kBinThreads == 4 * 32, "one warp per scanned quantity");
constexpr int kTotalsPerLane = kMaxChunks / 32;

struct GRef {
  double v[10];
  double gl_e, gl_mu;  // 1/2 + sin^2, -1/2 + sin^2
};

// Products of the couplings (eq. g_tilde), one per thread k < 10; nu_mu is
// unshifted.  Order: gLe^2 gLm^2 gLt^2 gRe^2 gRm^2 gRt^2 gLe.gRe gLm.gRm gLt.gRt
// kappa mu^2; delta mode: minus those of the reference point.
__device__ __forceinline__ void couplings(int k, const float* __restrict__ theta, double sin2w, double kappa,
                                          const GRef& gref, int delta, double* c) {
  if (k >= 10) return;
  // an SM sub-partition takes 64 cycles for any FP64 instruction of a warp, so
  // every thread picks its own two factors first and adds and multiplies once
  const double gl_e = gref.gl_e, gl_mu = gref.gl_mu;
  double x, y;
  if (k == 9) {
    x = kappa;
    y = (double)theta[4] * (double)theta[4];
  } else {
    const int kx = k < 6 ? k : k - 6, ky = k < 6 ? k : k - 3;  // gLe gLm gLt gRe gRm gRt
    const float tx = kx == 0 ? theta[0] : kx == 2 ? theta[2] : kx == 3 ? theta[1] : kx == 5 ? theta[3] : 0.f;
    const float ty = ky == 0 ? theta[0] : ky == 2 ? theta[2] : ky == 3 ? theta[1] : ky == 5 ? theta[3] : 0.f;
    x = (kx == 0 ? gl_e : kx < 3 ? gl_mu : sin2w) + (double)tx;
    y = (ky == 0 ? gl_e : ky < 3 ? gl_mu : sin2w) + (double)ty;
  }
  x *= y;
  if (delta) x -= gref.v[k];
  c[k] = x;
}

// A node's tables: {w P_e, w P_mu, w P_tau, w}, {1/E, clipped I0, I1, J, MM}
// and the bin that clips it; zeros beyond the last node.
struct Node {
  double w[4], q[5];
  int k;
};

__device__ __forceinline__ Node load_node(const ModelView& m, int n, int n_end) {
  Node d;
  const bool in = n < n_end;
  const size_t N = m.n_nodes;
#pragma unroll
  for (int k = 0; k < 4; ++k) d.w[k] = in ? m.node64[(k + 1) * N + n] : 0.0;
#pragma unroll
  for (int k = 0; k < 5; ++k) d.q[k] = in ? m.node_q[k * N + n] : 0.0;
  d.k = in ? m.node_k[n] : -1;
  return d;
}

// Prefix sums over the warp's 32 nodes (one per lane): X, Y, Z, V, and the
// clipped-bin terms over the nodes that end in the same bin.
struct Sums {
  double x, y, z, v, q;
};

// kPart 0: X, Y and V; 1: Z and the clipped terms; 2: all of them.  Only lanes
// below count need their sums.
template <int kPart>
__device__ __forceinline__ Sums scan_nodes(const Node& d, const double* c, int lane, int count = 32) {
  Sums s = {};
  const double r = d.q[0];
  const double a0 = fma(d.w[0], c[0], fma(d.w[1], c[1], d.w[2] * c[2]));
  const double a1 = fma(d.w[0], c[3], fma(d.w[1], c[4], d.w[2] * c[5]));
  const double a2 = fma(d.w[0], c[6], fma(d.w[1], c[7], d.w[2] * c[8])) * (kMe * r * r);  // times m_e / E^2
  const double v = d.w[3] * c[9], a1r = a1 * r;
  if (kPart != 1) {
    s.v = v;
    s.x = fma(-v, r, a0 + a1);
    s.y = fma(0.5, a2, a1r);
  }
  if (kPart != 0) {
    s.z = a1r * r;
    s.q = fma(a0, d.q[1], fma(a1, d.q[3], fma(-a2, d.q[2], v * d.q[4])));
  }
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    if (o >= count) break;
    if (kPart != 1) {
      const double px = __shfl_up_sync(0xffffffffu, s.x, o), py = __shfl_up_sync(0xffffffffu, s.y, o);
      const double pv = __shfl_up_sync(0xffffffffu, s.v, o);
      if (lane >= o) {
        s.x += px;
        s.y += py;
        s.v += pv;
      }
    }
    if (kPart != 0) {
      const double pz = __shfl_up_sync(0xffffffffu, s.z, o), pq = __shfl_up_sync(0xffffffffu, s.q, o);
      const int pk = __shfl_up_sync(0xffffffffu, d.k, o);
      if (lane >= o) {
        s.z += pz;
        if (pk == d.k) s.q += pq;
      }
    }
  }
  return s;
}

// Warp 0 takes X, Y and V of the chunk, warp 1 Z and the clipped terms: half
// the chain of FP64 instructions, on two sub-partitions.
__global__ void __launch_bounds__(64)
moments_kernel(ModelView m, const float* __restrict__ theta, double sin2w, double kappa, GRef gref, int delta,
               int chunk_nodes, double* __restrict__ totals, double* __restrict__ pre, double* __restrict__ clip) {
  __shared__ double cs[2][10];
  const int lane = threadIdx.x & 31, part = threadIdx.x >> 5;
  double* c = cs[part];
  const int n0 = blockIdx.x * chunk_nodes, n1 = min(m.n_nodes, n0 + chunk_nodes);
  Node next = load_node(m, n0 + lane, n1);  // ahead of the couplings
  couplings(lane, theta, sin2w, kappa, gref, delta, c);
  __syncwarp();
  double cx = 0.0, cy = 0.0, cz = 0.0, cv = 0.0;  // carry of the chunk's earlier tiles
  for (int base = n0; base < n1; base += 32) {
    const int n = base + lane;
    const bool more = base + 32 < n1;
    const Node d = next;
    if (more) next = load_node(m, n + 32, n1);
    if (part == 0) {
      Sums s = scan_nodes<0>(d, c, lane);
      if (base != n0) {
        s.x += cx;
        s.y += cy;
        s.v += cv;
      }
      if (n < n1) {
        pre[4 * (size_t)n] = s.x;
        pre[4 * (size_t)n + 1] = s.y;
        pre[4 * (size_t)n + 3] = s.v;
      }
      cx = more ? __shfl_sync(0xffffffffu, s.x, 31) : s.x;
      cy = more ? __shfl_sync(0xffffffffu, s.y, 31) : s.y;
      cv = more ? __shfl_sync(0xffffffffu, s.v, 31) : s.v;
    } else {
      Sums s = scan_nodes<1>(d, c, lane);
      if (base != n0) s.z += cz;
      if (n < n1) {
        pre[4 * (size_t)n + 2] = s.z;
        clip[n] = s.q;
      }
      cz = more ? __shfl_sync(0xffffffffu, s.z, 31) : s.z;
    }
  }
  // the dependents start here, not at the top: started early, they cost more than they hide
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (lane == 31) {
    double* t = totals + blockIdx.x;
    if (part == 0) {
      t[0] = cx;
      t[kMaxChunks] = cy;
      t[3 * kMaxChunks] = cv;
    } else {
      t[2 * kMaxChunks] = cz;
    }
  }
}

// Outputs (any may be null):
//   S_out[i]   = S_i(theta)
//   W_out[i]   = S_i(theta) / S_SM,i * E_SM,i   (E_SM,i where S_SM,i == 0)
//   ssm_out[i] = S_i(theta)                     (used once at create, theta = 0)
// kFew: at most kBinThreads nodes (a few lines): every block sums them itself,
// one tile of 32 a warp, and there is no first kernel (n_chunks tiles of 32).
// Otherwise totals, pre and clip are written by the grid this one waits for; they
// are not __restrict__: a load that may be taken for constant can move above the wait.
template <bool kFew>
__global__ void __launch_bounds__(kBinThreads)
bins_kernel(ModelView m, const float* theta, double sin2w, double kappa, GRef gref, int delta, int n_chunks,
            int chunk_nodes, const double* totals, const double2* pre, const double* clip, float* S_out, float* W_out,
            float* ssm_out) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  __shared__ double base[4][kFew ? 4 : kMaxChunks];  // sums of the chunks before this one, from its lane's first
  __shared__ double lbase[4][kFew ? 1 : 32];         // sums of the chunks before the lane's first
  __shared__ double sclip[kBinsPerBlock];
  __shared__ double2 spre[kFew ? 2 * kBinThreads : 1];
  __shared__ double sq[kFew ? kBinThreads : 1], c[kFew ? 10 : 1];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  // what does not depend on theta, ahead of the wait
  const int first = blockIdx.x * kBinsPerBlock;
  const int iq = first + t / kLanesPerBin, ib = first + t;
  const int2 nq = iq < m.n_t ? m.bin_n[iq] : make_int2(0, 0);
  int full = 0;
  double2 b0 = {0.0, 0.0}, b1 = {0.0, 0.0};
  float den = 0.f, esm = 0.f;
  if (t < kBinsPerBlock && ib < m.n_t) {
    full = m.bin_n[ib].x;
    b0 = m.bin_q[2 * (size_t)ib];
    b1 = m.bin_q[2 * (size_t)ib + 1];
    if (W_out) {
      den = m.ssm32[ib];
      esm = m.esm32[ib];
    }
  }
  double2 p0 = {0.0, 0.0}, p1 = {0.0, 0.0};
  if constexpr (kFew) {
    const Node d = load_node(m, t, m.n_nodes);
    couplings(t, theta, sin2w, kappa, gref, delta, c);
    __syncthreads();
    if (warp < n_chunks) {
      const Sums s = scan_nodes<2>(d, c, lane, m.n_nodes - 32 * warp);
      spre[2 * t] = make_double2(s.x, s.y);
      spre[2 * t + 1] = make_double2(s.z, s.v);
      sq[t] = s.q;
    }
    __syncthreads();
    if (t < 4) {
      double run = 0.0;
      for (int k = 0; k < n_chunks; ++k) {
        base[t][k] = run;
        const double2 e = spre[2 * min(32 * k + 31, m.n_nodes - 1) + t / 2];  // the tile's total
        run += t & 1 ? e.y : e.x;
      }
    }
    if (full > 0) {
      p0 = spre[2 * (full - 1)];
      p1 = spre[2 * (full - 1) + 1];
    }
    clip = sq;
  } else {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    double tot[kTotalsPerLane];
#pragma unroll
    for (int k = 0; k < kTotalsPerLane; ++k) {
      const int i = lane * kTotalsPerLane + k;
      tot[k] = i < n_chunks ? totals[warp * kMaxChunks + i] : 0.0;
    }
    if (full > 0) {  // t < kBinsPerBlock
      p0 = pre[2 * (size_t)(full - 1)];
      p1 = pre[2 * (size_t)(full - 1) + 1];
    }
    double run = tot[0];
    base[warp][lane * kTotalsPerLane] = 0.0;
#pragma unroll
    for (int k = 1; k < kTotalsPerLane; ++k) {
      base[warp][lane * kTotalsPerLane + k] = run;
      run += tot[k];
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double u = __shfl_up_sync(0xffffffffu, run, o);
      if (lane >= o) run += u;
    }
    run = __shfl_up_sync(0xffffffffu, run, 1);
    lbase[warp][lane] = lane == 0 ? 0.0 : run;
  }
  // clipped nodes [x, y) of the bin: the sums left at the last of them in each
  // tile of 32 nodes
  double q = 0.0;
  if (nq.x < nq.y) {
    for (int k = nq.x / 32 + t % kLanesPerBin; 32 * k < nq.y; k += 4 * kLanesPerBin) {
      double e[4];  // all in flight before the first is added
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = k + u * kLanesPerBin;
        e[u] = 32 * i < nq.y ? clip[min(nq.y, 32 * (i + 1)) - 1] : 0.0;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (32 * (k + u * kLanesPerBin) < nq.y) q += e[u];
    }
  }
#pragma unroll
  for (int o = kLanesPerBin / 2; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
  if (t % kLanesPerBin == 0) sclip[t / kLanesPerBin] = q;
  __syncthreads();
  if (t >= kBinsPerBlock || ib >= m.n_t) return;
  double v = sclip[t];
  if (full > 0) {
    const int k = (full - 1) / chunk_nodes;
    double X = base[0][k] + p0.x, Y = base[1][k] + p0.y, Z = base[2][k] + p1.x, V = base[3][k] + p1.y;
    if constexpr (!kFew) {
      const int l = k / kTotalsPerLane;
      X += lbase[0][l];
      Y += lbase[1][l];
      Z += lbase[2][l];
      V += lbase[3][l];
    }
    v += fma(b0.x, fma(b1.x, Z, fma(-b0.y, Y, X)), b1.y * V);
  }
  const float s = (float)v;
  if (S_out) S_out[ib] = s;
  if (ssm_out) ssm_out[ib] = s;
  // W = S/S_SM E_SM (E_SM where S_SM = 0); in delta mode S is the deviation
  // from the reference point and so is W (0 where S_SM = 0)
  if (W_out) W_out[ib] = den != 0.f ? (s / den) * esm : (delta ? 0.f : esm);
}

// ---------------------------------------------------------------------------
// Create-time helpers (FP64): S_SM, efficiency, lambda, E_SM and the
// pre-weighted basis shat_b,i = B_b,i E_SM,i / S_SM,i used by the batched
// path, where the weighted true spectrum of point p is
//   W_p,i = sum_b c_b(theta_p) shat_b,i = S_i(theta_p)/S_SM,i * E_SM,i.
// ---------------------------------------------------------------------------
__global__ void ssm_from_basis_kernel(const double* __restrict__ basis, int n_t, double gl_e, double gr_e,
                                      double gl_t, double gr_t, double* __restrict__ ssm) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_t) return;
  const double c[kNB] = {gl_e * gl_e, gr_e * gr_e, -gl_e * gr_e, gl_t * gl_t, gr_t * gr_t, -gl_t * gr_t, 1.0, 0.0};
  double s = 0.0;
#pragma unroll
  for (int b = 0; b < kNB; ++b) s += c[b] * basis[b * n_t + i];
  ssm[i] = s;
}

// Column sums eff_i = sum_j R_ji in FP64 (coalesced over i).
__global__ void efficiency_kernel(const float* __restrict__ R, int n_rec, int ld, int n_t, double* __restrict__ eff) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_t) return;
  double s = 0.0;
  for (int j = 0; j < n_rec; ++j) s += (double)R[(size_t)j * ld + i];
  eff[i] = s;
}

// lambda = exposure / sum_i eff_i S_SM,i (single block, fixed order).
__global__ void lambda_kernel(const double* __restrict__ eff, const double* __restrict__ ssm, int n_t,
                              double exposure, double* __restrict__ lambda_out) {
  __shared__ double red[32];
  double s = 0.0;
  for (int i = threadIdx.x; i < n_t; i += blockDim.x) s += eff[i] * ssm[i];
  s = warp_sum_d(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    *lambda_out = t > 0.0 ? exposure / t : 0.0;
  }
}

__global__ void esm_kernel(const double* __restrict__ ssm, const double* __restrict__ lambda, int n_t,
                           double* __restrict__ esm) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n_t) esm[i] = *lambda * ssm[i];
}

__global__ void shat_kernel(const double* __restrict__ basis, const double* __restrict__ ssm,
                            const double* __restrict__ esm, int n_t, int k_pad, float* __restrict__ shat,
                            float* __restrict__ shat_lo, float* __restrict__ esm32) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= k_pad) return;
  if (i >= n_t) {
#pragma unroll
    for (int b = 0; b < kNB; ++b) shat[b * k_pad + i] = shat_lo[b * k_pad + i] = 0.f;
    return;
  }
  const double s = ssm[i], e = esm[i];
  esm32[i] = (float)e;
#pragma unroll
  for (int b = 0; b < kNB; ++b) {
    double v;
    if (s != 0.0) v = basis[b * n_t + i] * (e / s);
    else v = (b == 6) ? e : 0.0;   // w_i = 1 where S_SM,i = 0
    const float hi = (float)v;
    shat[b * k_pad + i] = hi;
    shat_lo[b * k_pad + i] = (float)(v - (double)hi);
  }
}

// Weighted true spectrum of one point from the coefficient spectra (the
// recoil spectrum is a polynomial in the coupling monomials, Sec. II):
//   dW_i = sum_b (c_b(theta) - c_b(theta_ref)) shat_b,i
// with monomials and shat as hi + lo float pairs (delta = 0: the full W).
__global__ void weights_from_basis_kernel(const float* __restrict__ theta, dfloat sin2w, CoefRef cref,
                                          const float* __restrict__ shat, const float* __restrict__ shat_lo,
                                          int k_pad, float* __restrict__ W) {
  // a fold launched as this kernel's programmatic dependent may start now: it
  // streams R and waits for this grid's W before using it
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  __shared__ float ch[kNB], cl[kNB];
  if (threadIdx.x < kNB) {
    const dfloat s = sin2w;
    const dfloat gle = df_add(df_add(dfloat{0.5f, 0.f}, s), theta[0]), gre = df_add(s, theta[1]);
    const dfloat glt = df_add(df_add(dfloat{-0.5f, 0.f}, s), theta[2]), grt = df_add(s, theta[3]);
    const int b = threadIdx.x;
    dfloat c;
    if (b == 0) c = df_mul(gle, gle);
    else if (b == 1) c = df_mul(gre, gre);
    else if (b == 2) { c = df_mul(gle, gre); c = dfloat{-c.hi, -c.lo}; }
    else if (b == 3) c = df_mul(glt, glt);
    else if (b == 4) c = df_mul(grt, grt);
    else if (b == 5) { c = df_mul(glt, grt); c = dfloat{-c.hi, -c.lo}; }
    else if (b == 6) c = dfloat{1.f, 0.f};
    else c = two_prod(theta[4], theta[4]);
    const dfloat d = df_add(c, dfloat{-cref.hi[b], -cref.lo[b]});
    ch[b] = d.hi;
    cl[b] = d.lo;
  }
  __syncthreads();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= k_pad) return;
  float a = 0.f, t = 0.f;
#pragma unroll
  for (int b = 0; b < kNB; ++b) {
    const float sh = shat[(size_t)b * k_pad + i], sl = shat_lo[(size_t)b * k_pad + i];
    a = fmaf(ch[b], sh, a);
    t = fmaf(cl[b], sh, fmaf(ch[b], sl, t));
  }
  W[i] = a + t;
}

// Reference fold (create / set-reference time, FP64):
//   W_ref,i = sum_b c_b(theta_ref) B_b,i E_SM,i / S_SM,i   (E_SM,i where S_SM,i = 0)
//   mu_ref,j = sum_i R_ji W_ref,i
__global__ void wref_kernel(const double* __restrict__ basis, const double* __restrict__ ssm,
                            const double* __restrict__ esm, int n_t, CoefRef c, double* __restrict__ wref) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_t) return;
  const double sm = ssm[i], e = esm[i];
  if (sm == 0.0) {
    wref[i] = e;
    return;
  }
  double v = 0.0;
#pragma unroll
  for (int b = 0; b < kNB; ++b) v += ((double)c.hi[b] + (double)c.lo[b]) * basis[b * n_t + i];
  wref[i] = v * (e / sm);
}

__global__ void muref_kernel(const float* __restrict__ R, int ld, int n_t, const double* __restrict__ wref,
                             double* __restrict__ muref, float* __restrict__ muref32) {
  __shared__ double red[32];
  const int j = blockIdx.x;
  double s = 0.0;
  for (int i = threadIdx.x; i < n_t; i += blockDim.x) s += (double)R[(size_t)j * ld + i] * wref[i];
  s = warp_sum_d(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    muref[j] = t;
    muref32[j] = (float)t;
  }
}

}  // namespace

cudaError_t launch_reference_fold(srw_ctx* h, cudaStream_t s) {
  double* d_w = nullptr;
  cudaError_t e = dev_malloc_async(&d_w, sizeof(double) * h->n_t, s);
  if (e != cudaSuccess) return e;
  wref_kernel<<<(h->n_t + 255) / 256, 256, 0, s>>>(h->d_basis, h->d_ssm64, h->d_esm64, h->n_t, h->cref, d_w);
  muref_kernel<<<h->n_rec, 256, 0, s>>>(h->d_R, h->ld_r, h->n_t, d_w, h->d_muref64, h->d_muref32);
  if ((e = launch_result()) != cudaSuccess) return e;
  return cudaFreeAsync(d_w, s);
}

cudaError_t launch_weights_from_basis(const srw_ctx* h, const float* theta, float* W, cudaStream_t s) {
  weights_from_basis_kernel<<<(h->k_pad + 255) / 256, 256, 0, s>>>(theta, df_from_double(h->sin2w), h->cref,
                                                                  h->d_shat, h->d_shat_lo, h->k_pad, W);
  return launch_result();
}

cudaError_t launch_basis_fp64(const srw_ctx* h, cudaStream_t s) {
  const ModelView m = model_view(h);
  const double gl_mu = -0.5 + h->sin2w, gr_mu = h->sin2w;
  basis_fp64_kernel<<<h->n_t, kBasisThreads, 0, s>>>(m, gl_mu, gr_mu, h->kappa, h->d_basis);
  return launch_result();
}

cudaError_t launch_spectrum_point(const srw_ctx* h, const float* theta, float* S_out, float* W_out, float* ssm_out,
                                  cudaStream_t s, bool delta) {
  const ModelView m = model_view(h);
  GRef g;
  for (int k = 0; k < 10; ++k) g.v[k] = (double)h->gref[0][k] + (double)h->gref[1][k];
  g.gl_e = 0.5 + h->sin2w;
  g.gl_mu = -0.5 + h->sin2w;
  const int d = delta && h->use_ref ? 1 : 0;
  const int chunk = ((h->n_nodes - 1) / (32 * kMaxChunks) + 1) * 32, n_chunks = (h->n_nodes + chunk - 1) / chunk;
  double* totals = h->d_spec;
  double* pre = totals + 4 * kMaxChunks;
  double* clip = totals + 4 * kMaxChunks + 4 * (size_t)h->n_nodes;
  const int grid = (h->n_t + kBinsPerBlock - 1) / kBinsPerBlock;
  if (h->n_nodes <= kBinThreads) {
    bins_kernel<true><<<grid, kBinThreads, 0, s>>>(m, theta, h->sin2w, h->kappa, g, d, n_chunks, 32, nullptr, nullptr,
                                                   nullptr, S_out, W_out, ssm_out);
    return launch_result();
  }
  moments_kernel<<<n_chunks, 64, 0, s>>>(m, theta, h->sin2w, h->kappa, g, d, chunk, totals, pre, clip);
  cudaError_t e = launch_result();
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kBinThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, bins_kernel<false>, m, theta, h->sin2w, h->kappa, g, d, n_chunks, chunk,
                         (const double*)totals, reinterpret_cast<const double2*>(pre), (const double*)clip, S_out, W_out, ssm_out);
  return e != cudaSuccess ? e : launch_result();
}

// Builds S_SM (FP64), lambda, E_SM and shat.  Requires d_basis.
cudaError_t launch_build_shat(srw_ctx* h, cudaStream_t s) {
  const int n_t = h->n_t, thr = 256;
  const int g_t = (n_t + thr - 1) / thr;
  const double s2 = h->sin2w;
  ssm_from_basis_kernel<<<g_t, thr, 0, s>>>(h->d_basis, n_t, 0.5 + s2, s2, -0.5 + s2, s2, h->d_ssm64);
  cudaError_t e = launch_result();
  if (e != cudaSuccess) return e;
  if (!h->has_esm_input) {
    double* d_eff = nullptr;
    double* d_lam = nullptr;
    if ((e = dev_malloc_async(&d_eff, sizeof(double) * (n_t + 1), s)) != cudaSuccess) return e;
    d_lam = d_eff + n_t;
    efficiency_kernel<<<g_t, thr, 0, s>>>(h->d_R, h->n_rec, h->ld_r, n_t, d_eff);
    lambda_kernel<<<1, 1024, 0, s>>>(d_eff, h->d_ssm64, n_t, h->exposure, d_lam);
    esm_kernel<<<g_t, thr, 0, s>>>(h->d_ssm64, d_lam, n_t, h->d_esm64);
    if ((e = launch_result()) != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(&h->lambda, d_lam, sizeof(double), cudaMemcpyDeviceToHost, s)) != cudaSuccess) return e;
    if ((e = cudaFreeAsync(d_eff, s)) != cudaSuccess) return e;
  }
  const int g_k = (h->k_pad + thr - 1) / thr;
  shat_kernel<<<g_k, thr, 0, s>>>(h->d_basis, h->d_ssm64, h->d_esm64, n_t, h->k_pad, h->d_shat, h->d_shat_lo,
                                    h->d_esm32);
  return launch_result();
}

}  // namespace srw
