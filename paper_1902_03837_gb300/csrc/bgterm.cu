// Bruneval-Gonze extrapolar correction (X-terminator): Eq. (X_term_def) and
// Appendix C (Eqs. rhotw-term, F-term, X-term).  The bands left out of the
// sum get one energy eps_bar and no occupation; by the closure relation over
// all bands at k,
//
//   sum_{n >= nb} rho_nm(G) conj(rho_nm(G'))
//       = rho~_{m,k-q}(G - G') - sum_{n < nb} rho_nm(G) conj(rho_nm(G')),
//
// so the corrected chi0 is the contraction over every band n < nb with the
// weights w_t - wbar_m (done by the weights kernel and the usual contraction)
// plus sum_{k', m} wbar_{mk'}(w) rho~_{mk'}(G - G').  The diagonal densities
// rho~ come from the rho kernel in its same-band mode on the set of
// difference vectors d = G_i - G_j; the two kernels here form that last term.
#include "internal.cuh"

namespace chi0 {

namespace {

// P[iw][d] for 32 vectors d per block and up to eight frequencies: eight warps
// take every eighth state and add up (one thread per (d, frequency) walked over
// all states, one load after the other).  Bound by the FP64 units, to which the
// conversions of an FP32 density belong: each is converted once for the eight
// frequencies (768 states, 1760 vectors, 16 frequencies 217 -> 159 us).
constexpr int kBgW = 8, kBgF = 8;
template <typename TOUT>
__global__ void __launch_bounds__(32 * kBgW)
k_bg_sum(const TOUT* __restrict__ rd, const BgChunks ch, const double* __restrict__ wbar, int64_t ntd,
         int nd, int nw, double2* __restrict__ P) {
  __shared__ double2 sums[kBgW][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int d = blockIdx.x * 32 + lane;
  const int iw0 = blockIdx.y * kBgF, nf = min(kBgF, nw - iw0);
  const double* w = wbar + (size_t)iw0 * ntd;
  double2 s[kBgF];
#pragma unroll
  for (int f = 0; f < kBgF; ++f) s[f] = make_double2(0.0, 0.0);
  if (d < nd) {
    int c = 0;
    while (c + 1 < ch.n && d >= ch.start[c + 1]) ++c;
    const int64_t stride = ch.start[c + 1] - ch.start[c];
    const TOUT* p = rd + ch.off[c] + (d - ch.start[c]);
#pragma unroll 2
    for (int64_t t = warp; t < ntd; t += kBgW) {
      const TOUT v = p[t * stride];
      const double vx = (double)v.x, vy = (double)v.y;
#pragma unroll
      for (int f = 0; f < kBgF; ++f) {
        if (f < nf) {
          const double wt = w[(size_t)f * ntd + t];
          s[f].x = fma(wt, vx, s[f].x);
          s[f].y = fma(wt, vy, s[f].y);
        }
      }
    }
  }
#pragma unroll
  for (int f = 0; f < kBgF; ++f) {
    if (f >= nf) break;
    sums[warp][lane] = s[f];
    __syncthreads();
    if (warp == 0 && d < nd) {
      double2 a = s[f];
      for (int q = 1; q < kBgW; ++q) {
        a.x += sums[q][lane].x;
        a.y += sums[q][lane].y;
      }
      P[(size_t)(iw0 + f) * nd + d] = a;
    }
    __syncthreads();
  }
}

// chi[iw][i][j] += v, chi[iw][j][i] += conj(v) for i >= j, with
// v = (P[d_ij] + conj(P[d_ji])) / 2 (exactly Hermitian; real on the diagonal)
// imag = 1 adds i times the Hermitised term (the imaginary parts of complex
// weights, added to a full complex chi0 of a real-axis frequency)
__global__ void k_bg_apply(const double2* __restrict__ P, const int32_t* __restrict__ didx, int ng, int nd,
                           double2* __restrict__ chi, int imag) {
  const int iw = blockIdx.y;
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)ng * ng) return;
  const int i = (int)(e / ng), j = (int)(e % ng);
  if (i < j) return;
  const double2* Pw = P + (size_t)iw * nd;
  const double2 a = Pw[didx[(size_t)i * ng + j]], b = Pw[didx[(size_t)j * ng + i]];
  double vx = 0.5 * (a.x + b.x), vy = 0.5 * (a.y - b.y);
  double2* cw = chi + (size_t)iw * ng * ng;
  if (i == j) vy = 0.0;
  // lower entry += v, upper entry += conj(v); times i when imag
  const double2 lo = imag ? make_double2(-vy, vx) : make_double2(vx, vy);
  const double2 up = imag ? make_double2(vy, vx) : make_double2(vx, -vy);
  double2 x = cw[(size_t)i * ng + j];
  cw[(size_t)i * ng + j] = make_double2(x.x + lo.x, x.y + lo.y);
  if (i != j) {
    x = cw[(size_t)j * ng + i];
    cw[(size_t)j * ng + i] = make_double2(x.x + up.x, x.y + up.y);
  }
}

}  // namespace

template <typename TOUT>
cudaError_t launch_bg_sum(const TOUT* rd, const BgChunks& ch, const double* wbar, int64_t ntd, int nd,
                          int nw, double2* P, cudaStream_t s) {
  if (nd <= 0 || nw <= 0) return cudaSuccess;
  k_bg_sum<TOUT><<<dim3((unsigned)((nd + 31) / 32), (unsigned)((nw + kBgF - 1) / kBgF)), 32 * kBgW, 0, s>>>(
      rd, ch, wbar, ntd, nd, nw, P);
  return cudaGetLastError();
}

cudaError_t launch_bg_apply(const double2* P, const int32_t* didx, int ng, int nd, int nw, double2* chi,
                            cudaStream_t s, int imag) {
  if (ng <= 0 || nw <= 0) return cudaSuccess;
  const int64_t n = (int64_t)ng * ng;
  k_bg_apply<<<dim3((unsigned)((n + 255) / 256), (unsigned)nw), 256, 0, s>>>(P, didx, ng, nd, chi, imag);
  return cudaGetLastError();
}

template cudaError_t launch_bg_sum<float2>(const float2*, const BgChunks&, const double*, int64_t, int, int,
                                           double2*, cudaStream_t);
template cudaError_t launch_bg_sum<double2>(const double2*, const BgChunks&, const double*, int64_t, int, int,
                                            double2*, cudaStream_t);

}  // namespace chi0
