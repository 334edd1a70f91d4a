// Batched fold in FP32 on the SIMT pipes (the FP32 way of the batched scan).
//
// For P parameter points the fold of eq. matrix_reweight becomes the
// contraction  M[p][j] = sum_i W[p][i] R[j][i]  with the reweighted true
// spectra W[p][i] = w_i(theta_p) E_SM,i.  Because the recoil spectrum is a
// polynomial in the couplings, W[p][i] = sum_b c_b(theta_p) shat_b,i with the
// eight pre-weighted coefficient spectra shat (built once in FP64); each
// block produces its W tile on chip from shat and the 8 coefficients of its
// points, so W is never written to memory.  The epilogue adds the summed
// background, applies the mask, evaluates the Poisson terms and reduces over
// its rec bins per point into FP64 partials (one per 64 bins).  The fold is
// taken of W(theta) - W_ref; the FP64 reference fold R W_ref enters with the
// background (b64 argument = background + reference fold).
//
// Accumulation: FP32 FMAs over one 16-wide K tile, tiles combined with Kahan
// compensation.  The rounding of an FMA chain is not independent from row to
// row: neighbouring reconstructed bins accumulate nearly the same sequence of
// partial sums, so their errors share a sign, and -2 ln L sums them with the
// weights 1 - n_j/mu_j, which share it too near a shifted spectrum.  The
// error of a chain grows with its length; 64-term chains moved -2 ln L by
// 1.7e-4 at a point 220 units from the data (FP32 emulation and GB300 agree),
// 16-term chains by 2e-5.

#include <algorithm>
#include <vector>

#include "dfloat.cuh"
#include "f32x2.cuh"
#include "poisson.cuh"
#include "srw_internal.h"

namespace srw {
namespace {

constexpr int kTile = 128;  // rec bins per tile of the transposed response copy
constexpr int BK = 16;      // true bins per K tile (and per FMA chain)
constexpr int THR = 128;
constexpr int kRing = 4;    // K tiles of R in flight or in use
constexpr int kNC = kNB - 1;  // monomials of a point's deviation (the constant one is always in the reference)

// Thread block: MI x NI groups of 4 points x 4 rec bins a thread, a warp 8 x 4
// lanes of them, four warps side by side along the bins.
//   <2, 2>: 64 points x 128 bins.  A thread's 8 x 8 outputs take four 128-bit
//           shared loads per 64 FMAs, half of the 4 x 8 outputs' six, which
//           kept the kernel at the shared-memory limit (26 % of the FP32 rate);
//           with 255 registers two blocks of four warps share an SM, and the
//           one's epilogue and W production run beside the other's FMAs.
//   <1, 1>: 32 points x 64 bins, for grids of fewer large tiles than SMs.
template <int MI, int NI>
struct SimtShape {
  static constexpr int BM = MI * 32, BN = NI * 64;
  static constexpr int kRow = BN + 16;  // floats per true bin of a ring slot: R, then the 14 spectra values (16)
  static constexpr int kWPer = BM * BK / THR;  // W elements a thread forms per K tile
};

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Coupling monomials c_b(theta) (see srw_internal.h) in double-float
// arithmetic, returned as hi + lo float pairs so that W carries no per-theta
// rounding bias.
__device__ __forceinline__ void coefficients(const float* th, dfloat s, const CoefRef& ref, float* hi, float* lo) {
  const dfloat gle = df_add(df_add(dfloat{0.5f, 0.f}, s), th[0]), gre = df_add(s, th[1]);
  const dfloat glt = df_add(df_add(dfloat{-0.5f, 0.f}, s), th[2]), grt = df_add(s, th[3]);
  const dfloat x = df_mul(gle, gre), y = df_mul(glt, grt);
  const dfloat c[kNB] = {df_mul(gle, gle), df_mul(gre, gre), {-x.hi, -x.lo}, df_mul(glt, glt),
                         df_mul(grt, grt), {-y.hi, -y.lo}, {1.f, 0.f}, two_prod(th[4], th[4])};
#pragma unroll
  for (int b = 0; b < kNB; ++b) {
    if (b == 6) continue;
    const dfloat d = df_add(c[b], dfloat{-ref.hi[b], -ref.lo[b]});  // deviation from the reference point
    hi[b < 6 ? b : 6] = d.hi;
    lo[b < 6 ? b : 6] = d.lo;
  }
}

// R is read from a copy laid out for this kernel at create, Rt[tile of 128
// bins][true bin][bin], and the spectra from shk[true bin][16] (seven hi, pad,
// seven lo, pad): a K tile is then rows of contiguous floats that asynchronous
// 16-byte copies bring in three K tiles ahead (the row-major R went through
// registers and was transposed by four 4-byte stores per load).  order: {first
// and end K tile holding nonzero response, rec tile, 0}, longest range first,
// so that the last wave holds the short ones.  K tiles of zeros more or less
// (128 bins have a longer range than 64) do not change a bin's value: with a
// sum x of 0 a step of the Kahan sum sends (s, c) to t = fl(s - c) and
// (t - s) + c, and as |c| is at most a few units in the last place of s, that
// difference is exact: t minus the new c is s - c, which is all that is read.
template <int MI, int NI>
__global__ void __launch_bounds__(THR, MI * NI == 4 ? 2 : 4)
fold_simt_kernel(const float* __restrict__ theta, int P, dfloat sin2w, CoefRef cref, const float* __restrict__ shk,
                 int k_pad, const float* __restrict__ Rt, int n_rec, const float4* __restrict__ consts,
                 const double* __restrict__ n64, const double* __restrict__ b64, double* __restrict__ parts,
                 float* __restrict__ musig_out, const float* __restrict__ muref, unsigned* __restrict__ status,
                 const int4* __restrict__ order) {
  using S = SimtShape<MI, NI>;
  constexpr int BM = S::BM, BN = S::BN;
  __shared__ __align__(16) float ring[kRing][BK][S::kRow];
  __shared__ __align__(16) float Ws[2][BK][BM];
  __shared__ float cs[2 * kNC][BM];

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, lm = lane >> 2, ln = lane & 3;
  const int m0 = blockIdx.x * BM;
  const int4 od = order[blockIdx.y];
  const int2 kr = make_int2(od.x, od.y);
  const int j0 = od.z * BN;  // first rec bin

  for (int r = tid; r < BM; r += THR) {
    float hi[kNC], lo[kNC];
    if (m0 + r < P) {
      coefficients(theta + (size_t)(m0 + r) * 5, sin2w, cref, hi, lo);
    } else {
#pragma unroll
      for (int b = 0; b < kNC; ++b) hi[b] = lo[b] = 0.f;
    }
#pragma unroll
    for (int b = 0; b < kNC; ++b) {
      cs[b][r] = hi[b];
      cs[kNC + b][r] = lo[b];
    }
  }

  const float* Rtile = Rt + (size_t)(j0 / kTile) * k_pad * kTile + (j0 % kTile);
  auto load_tile = [&](int kt) {
    if (kt < kr.y) {
      SRW_CHECK(status, kt >= 0 && (kt + 1) * BK <= k_pad);
      float(*dst)[S::kRow] = ring[(kt - kr.x) % kRing];
#pragma unroll
      for (int q = tid; q < BK * BN / 4; q += THR) {
        const int k = q / (BN / 4), c = (q % (BN / 4)) * 4;
        cp_async16(&dst[k][c], Rtile + (size_t)(kt * BK + k) * kTile + c);
      }
      if (tid < BK * 4)
        cp_async16(&dst[tid >> 2][BN + (tid & 3) * 4], shk + (size_t)(kt * BK + (tid >> 2)) * 16 + (tid & 3) * 4);
    }
    cp_async_commit();  // one group per K tile, empty past the end
  };
  // W^T tile: W[p][k] = sum_b c_b(p) shat_b[k], (c_hi + c_lo)(s_hi + s_lo) without lo*lo
  auto make_w = [&](int kt) {
    const float(*src)[S::kRow] = ring[(kt - kr.x) % kRing];
    float(*dst)[BM] = Ws[(kt - kr.x) & 1];
    const int p = tid % BM, kb = tid / BM * S::kWPer;
    float ch[kNC], cl[kNC];
#pragma unroll
    for (int b = 0; b < kNC; ++b) {
      ch[b] = cs[b][p];
      cl[b] = cs[kNC + b][p];
    }
#pragma unroll 2
    for (int k = kb; k < kb + S::kWPer; ++k) {
      const float4* q = reinterpret_cast<const float4*>(&src[k][BN]);
      const float4 h0 = q[0], h1 = q[1], l0 = q[2], l1 = q[3];
      const float sh[kNC] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z};
      const float sl[kNC] = {l0.x, l0.y, l0.z, l0.w, l1.x, l1.y, l1.z};
      float s = 0.f, t = 0.f;
#pragma unroll
      for (int b = 0; b < kNC; ++b) {
        s = fmaf(ch[b], sh[b], s);
        t = fmaf(cl[b], sh[b], fmaf(ch[b], sl[b], t));
      }
      dst[k][p] = s + t;
    }
  };

  // packed along the bins: pair c of point row r holds bins 2c, 2c + 1 of the thread's 4 NI
  uint64_t sum[4 * MI][2 * NI], comp[4 * MI][2 * NI];
#pragma unroll
  for (int r = 0; r < 4 * MI; ++r)
#pragma unroll
    for (int c = 0; c < 2 * NI; ++c) sum[r][c] = comp[r][c] = 0ull;

#pragma unroll
  for (int q = 0; q < kRing - 1; ++q) load_tile(kr.x + q);
  cp_async_wait<kRing - 2>();
  __syncthreads();  // the first K tile and the coefficients
  if (kr.x < kr.y) make_w(kr.x);
  for (int kt = kr.x; kt < kr.y; ++kt) {
    cp_async_wait<kRing - 3>();  // this thread's copies of K tile kt + 1
    __syncthreads();             // everybody's, W of kt, and the end of kt - 1
    load_tile(kt + kRing - 1);   // into the slot of kt - 1
    const float(*rs)[S::kRow] = ring[(kt - kr.x) % kRing];
    const float(*ws)[BM] = Ws[(kt - kr.x) & 1];
    uint64_t acc[4 * MI][2 * NI];
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      float a[4 * MI];
      uint64_t b[2 * NI];
#pragma unroll
      for (int i = 0; i < MI; ++i) {
        const float4 v = *reinterpret_cast<const float4*>(&ws[k][i * 32 + lm * 4]);
        a[4 * i] = v.x; a[4 * i + 1] = v.y; a[4 * i + 2] = v.z; a[4 * i + 3] = v.w;
      }
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&rs[k][warp * (16 * NI) + i * 16 + ln * 4]);
        b[2 * i] = v.x;
        b[2 * i + 1] = v.y;
      }
#pragma unroll
      for (int r = 0; r < 4 * MI; ++r) {
        const uint64_t aa = pk(a[r], a[r]);
#pragma unroll
        for (int c = 0; c < 2 * NI; ++c) acc[r][c] = k == 0 ? mul2(aa, b[c]) : fma2(aa, b[c], acc[r][c]);
      }
    }
    // each 16-term chain is added to the running sum with Kahan compensation
#pragma unroll
    for (int r = 0; r < 4 * MI; ++r)
#pragma unroll
      for (int c = 0; c < 2 * NI; ++c) {
        const uint64_t y = sub2(acc[r][c], comp[r][c]);
        const uint64_t t = add2(sum[r][c], y);
        comp[r][c] = sub2(sub2(t, sum[r][c]), y);
        sum[r][c] = t;
      }
    if (kt + 1 < kr.y) make_w(kt + 1);
  }
  cp_async_wait<0>();

  const int jw = j0 + warp * (16 * NI) + ln * 4;  // bins jw + 16 i + 0..3
  if (musig_out != nullptr) {  // batched folded spectra: deviation + reference fold
#pragma unroll
    for (int i = 0; i < NI; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int j = jw + 16 * i + c;
        if (j >= n_rec) continue;
        const float ref = __ldg(muref + j);
#pragma unroll
        for (int r = 0; r < 4 * MI; ++r) {
          const int p = m0 + (r / 4) * 32 + lm * 4 + (r & 3);
          const float2 s2 = unpk(sum[r][2 * i + c / 2]), c2 = unpk(comp[r][2 * i + c / 2]);
          const float v = (c & 1) ? s2.y - c2.y : s2.x - c2.x;
          if (p < P) musig_out[(size_t)p * n_rec + j] = v + ref;
        }
      }
  }
  if (parts == nullptr) return;
  // Epilogue: Poisson terms over this block's rec bins per point, in double-
  // float: FP64 (a warp's instruction takes the SM's unit 16 cycles) spent
  // 0.7 ms of a 4096-point call's 2.7 ms on the logarithms here.  A sum over 16
  // bins (four a thread, then its four neighbours) is in double-float, the four
  // of 64 bins are added in FP64 in the order of the bins and are one partial
  // sum: the same in every tile shape, so that a point's value does not depend
  // on the batch that holds it.
  // the ring is free (its last copies landed above)
  float2(*psum)[BM] = reinterpret_cast<float2(*)[BM]>(&ring[0][0][0]);  // [16 bins][point]
  int(*pinf)[BM] = reinterpret_cast<int(*)[BM]>(&ring[1][0][0]);
  static_assert(sizeof(float2) * 4 * NI * BM <= sizeof(ring[0]), "sums of four warps in a ring slot");
  __syncthreads();
#pragma unroll
  for (int i = 0; i < NI; ++i) {
    dfloat d[4 * MI];
    bool inf[4 * MI];
#pragma unroll
    for (int r = 0; r < 4 * MI; ++r) {
      d[r] = {0.f, 0.f};
      inf[r] = false;
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int j = jw + 16 * i + c;
      if (j >= n_rec) continue;
      const float4 nb = __ldg(consts + 2 * j), mk = __ldg(consts + 2 * j + 1);  // {n, n lo, b, b lo}, {mask, ...}
      if (mk.x == 0.f) continue;
#pragma unroll
      for (int r = 0; r < 4 * MI; ++r) {
        const float2 s2 = unpk(sum[r][2 * i + c / 2]), c2 = unpk(comp[r][2 * i + c / 2]);
        const dfloat dev = two_sum((c & 1) ? s2.y : s2.x, (c & 1) ? -c2.y : -c2.x);
        dfloat t;
        if (!poisson_term_df(df_add(dev, dfloat{nb.z, nb.w}), dfloat{nb.x, nb.y}, &t)) {
          const double x = poisson_term_f64(((double)dev.hi + (double)dev.lo) + b64[j], n64[j]);
          t = isfinite(x) ? df_from_double(x) : dfloat{(float)x, 0.f};
        }
        if (isinf(t.hi)) inf[r] = true;
        else d[r] = df_add(d[r], t);
      }
    }
#pragma unroll
    for (int r = 0; r < 4 * MI; ++r) {
#pragma unroll
      for (int o = 1; o <= 2; o <<= 1) {
        d[r] = df_add(d[r], df_shfl_xor(d[r], o));
        inf[r] = __shfl_xor_sync(0xffffffffu, (int)inf[r], o) || inf[r];
      }
      if (ln == 0) {
        const int q = (r / 4) * 32 + lm * 4 + (r & 3);
        psum[warp * NI + i][q] = make_float2(d[r].hi, d[r].lo);
        pinf[warp * NI + i][q] = inf[r];
      }
    }
  }
  __syncthreads();
  for (int x = tid; x < NI * BM; x += THR) {
    const int q = x % BM, u = x / BM;  // 64 bins from j0 + 64 u on
    if (m0 + q >= P || j0 + 64 * u >= n_rec) continue;
    double s = 0.0;
    bool any = false;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      s += (double)psum[4 * u + w][q].x + (double)psum[4 * u + w][q].y;
      any |= pinf[4 * u + w][q] != 0;
    }
    parts[(size_t)(od.z * NI + u) * P + m0 + q] = any ? __longlong_as_double(0x7ff0000000000000LL) : s;
  }
}

// Rt[tile][k][128] from the row-major R (zero beyond n_rec), and shk[k][16].
// One block per 32 x 32 elements in one grid dimension (the others end at 65,535).
__global__ void simt_layout_kernel(const float* __restrict__ R, int n_rec, int ld, int k_pad,
                                   float* __restrict__ Rt) {
  __shared__ float s[32][33];
  const int k0 = (int)(blockIdx.x % (k_pad / 32)) * 32, r0 = (int)(blockIdx.x / (k_pad / 32)) * 32;
  for (int i = threadIdx.y; i < 32; i += 8) {
    const int j = r0 + i, k = k0 + threadIdx.x;
    s[i][threadIdx.x] = j < n_rec && k < ld ? R[(size_t)j * ld + k] : 0.f;
  }
  __syncthreads();
  const int t = r0 / kTile;
  for (int i = threadIdx.y; i < 32; i += 8)
    Rt[((size_t)t * k_pad + k0 + i) * kTile + r0 % kTile + threadIdx.x] = s[threadIdx.x][i];
}
__global__ void simt_spectra_kernel(const float* __restrict__ shat, const float* __restrict__ shat_lo, int k_pad,
                                    float* __restrict__ shk) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= k_pad) return;
#pragma unroll
  for (int b = 0; b < kNC; ++b) {
    const int src = b < 6 ? b : 7;
    shk[(size_t)k * 16 + b] = shat[(size_t)src * k_pad + k];
    shk[(size_t)k * 16 + 8 + b] = shat_lo[(size_t)src * k_pad + k];
  }
  shk[(size_t)k * 16 + 7] = shk[(size_t)k * 16 + 15] = 0.f;
}

template <int MI, int NI>
void launch_shape(const srw_ctx* h, const float* theta, int P, double* parts, cudaStream_t s, float* musig_out,
                  const int4* order) {
  using S = SimtShape<MI, NI>;
  const dim3 grid((P + S::BM - 1) / S::BM, (h->n_rec + S::BN - 1) / S::BN);
  fold_simt_kernel<MI, NI><<<grid, THR, 0, s>>>(theta, P, df_from_double(h->sin2w), h->cref, h->d_simt_sh, h->k_pad,
                                                h->d_simt_r, h->n_rec, h->d_simt_c, h->d_n64, h->d_bref64, parts,
                                                musig_out, h->d_muref32, h->d_status, order);
}

// The small tile where the large ones do not give every SM a block.
bool small_tile(const srw_ctx* h, int P) {
  const long long blocks = ((P + 63LL) / 64) * ((h->n_rec + 127) / 128);
  return blocks < h->sm_count;
}

}  // namespace

int fold_simt_parts(int n_rec) { return (n_rec + 63) / 64; }

cudaError_t launch_fold_simt(const srw_ctx* h, const float* theta, int P, double* parts, cudaStream_t s,
                             int* n_parts, float* musig_out) {
  if (small_tile(h, P)) launch_shape<1, 1>(h, theta, P, parts, s, musig_out, h->d_simt_kr + (h->n_rec + 127) / 128);
  else launch_shape<2, 2>(h, theta, P, parts, s, musig_out, h->d_simt_kr);
  if (n_parts) *n_parts = fold_simt_parts(h->n_rec);
  return launch_result();
}

// Per rec tile of 128 and of 64 bins the K tiles [first, end) between its
// first and last nonzero column of R (FP32, exact zeros outside; a tile
// without any nonzero element gets an empty range), longest first; and the
// copies of simt_ready.
cudaError_t simt_prepare(srw_ctx* h, const std::vector<float>& R, cudaStream_t s) {
  const int n_kt = h->k_pad / BK, cols = std::min(h->ld_r, h->k_pad);
  std::vector<int4> kr;
  for (int bn = 128; bn >= 64; bn -= 64) {
    const size_t first_of = kr.size();
    for (int t = 0; t * bn < h->n_rec; ++t) {
      int first = cols, last = -1;
      for (int j = t * bn; j < std::min(h->n_rec, (t + 1) * bn); ++j) {
        const float* row = R.data() + (size_t)j * h->ld_r;
        for (int k = 0; k < first; ++k)
          if (row[k] != 0.f) {
            first = k;
            break;
          }
        for (int k = cols - 1; k > last; --k)
          if (row[k] != 0.f) {
            last = k;
            break;
          }
      }
      kr.push_back(last < 0 ? make_int4(0, 0, t, 0) : make_int4(first / BK, std::min(n_kt, last / BK + 1), t, 0));
    }
    std::stable_sort(kr.begin() + first_of, kr.end(),
                     [](const int4& a, const int4& b) { return a.y - a.x > b.y - b.x; });
  }
  cudaError_t e = cudaSuccess;
  if (!h->d_simt_kr && (e = dev_malloc(&h->d_simt_kr, sizeof(int4) * kr.size())) != cudaSuccess) return e;
  h->device_bytes += sizeof(int4) * kr.size();
  e = cudaMemcpyAsync(h->d_simt_kr, kr.data(), sizeof(int4) * kr.size(), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return e;
  e = simt_ready(h);
  return e == cudaErrorMemoryAllocation ? cudaSuccess : e;  // only the FP32 batch reads the copies: it tries again
}

// The kernel's copies of R (as large as R) and of the coefficient spectra,
// made with the handle, or by the first FP32 batch where there was no room.
cudaError_t simt_ready(srw_ctx* h) {
  if (h->d_simt_r && h->d_simt_sh) return cudaSuccess;
  const int nt = (h->n_rec + kTile - 1) / kTile;
  const size_t bytes[2] = {sizeof(float) * (size_t)nt * kTile * h->k_pad, sizeof(float) * 16 * (size_t)h->k_pad};
  cudaStream_t s = h->own_stream;
  float *r = nullptr, *sh = nullptr;
  cudaError_t e = dev_malloc(&sh, bytes[1]);
  if (e == cudaSuccess) e = dev_malloc(&r, bytes[0]);
  if (e == cudaSuccess) {
    simt_layout_kernel<<<(unsigned)nt * (kTile / 32) * (h->k_pad / 32), dim3(32, 8), 0, s>>>(h->d_R, h->n_rec, h->ld_r,
                                                                                             h->k_pad, r);
    simt_spectra_kernel<<<(h->k_pad + 255) / 256, 256, 0, s>>>(h->d_shat, h->d_shat_lo, h->k_pad, sh);
    e = launch_result();
    const cudaError_t es = cudaStreamSynchronize(s);
    if (e == cudaSuccess) e = es;
  }
  if (e != cudaSuccess) {
    if (r) cudaFree(r);
    if (sh) cudaFree(sh);
    cudaGetLastError();  // a failed allocation is not the next launch's error
    return e;
  }
  h->d_simt_r = r;
  h->d_simt_sh = sh;
  h->device_bytes += bytes[0] + bytes[1];
  return cudaSuccess;
}

}  // namespace srw
