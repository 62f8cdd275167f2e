// Transition weights and the FP64 form of the chi0 contraction.
//
// Appendix B of the paper writes chi0 as frequency factors F_{nmk}(w) times
// frequency-independent products R^{nmk}_{GG'} = f_s/(N_k Omega) x (occupation
// factor) x rho rho^* (Eqs. X_IP_split, X_IP_split1, X_IP_split2).  Here the
// occupation factor, prefactor and two-pole frequency factor of each
// transition are folded into one real weight per (w, t), and
//
//     chi0(w) = sum_t w_t(w) rho_t rho_t^H   (Hermitian),
//
// is accumulated over bounded transition chunks (the paper's reduction over
// the k/c/v distribution becomes an on-device sum of chunk partials).
#include <algorithm>

#include "internal.cuh"

namespace chi0 {

namespace {

// w_t = pref (f_m - f_n) [1/(z + D) - 1/(z - D)] with z = w + i eta purely
// imaginary (z = i s): the bracket is 2 D / (D^2 + s^2), real.
// Frequency factor of one transition with energy difference d = e_m - e_n:
//   1/(w + d + i eta) - 1/(w - d + i eta)
// kind 0: w = i om (imaginary axis; the factor is real, 2d/(d^2 + (om+eta)^2));
// kind 1 / 2: w = om on the real axis, the real / imaginary part.
__device__ __forceinline__ double pole_weight(int kind, double om, double eta, double d) {
  if (kind == 0) {
    const double sw = om + eta;
    const double den = d * d + sw * sw;
    return den > 0.0 ? 2.0 * d / den : 0.0;
  }
  const double a = om + d, b = om - d;
  const double da = a * a + eta * eta, db = b * b + eta * eta;
  if (!(da > 0.0) || !(db > 0.0)) return 0.0;
  return kind == 1 ? a / da - b / db : eta / db - eta / da;
}

__global__ void k_weights(int nk, int n_lo, int Nn, int Nm, int nb, const int32_t* __restrict__ kq,
                          const double* __restrict__ eps, const double* __restrict__ occ,
                          const double* __restrict__ omega_im, const int* __restrict__ vkind, int nw,
                          double eta, double pref, double occ_tol, int bg, double eps_bar,
                          const double* __restrict__ dpole, const double* __restrict__ epsd, int nd,
                          double* __restrict__ w, int k0, const int64_t* __restrict__ perm, int64_t nrow) {
  const int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= nrow) return;
  const int64_t t = perm ? perm[row] : row;
  const int m = (int)(t % Nm);
  const int64_t r = t / Nm;
  const int n = n_lo + (int)(r % Nn);
  const int ik = k0 + (int)(r / Nn);   // global k (the transitions cover k0 .. k0 + nk - 1)
  const int ikp = kq[ik];
  const double df = occ[(size_t)ikp * nb + m] - occ[(size_t)ik * nb + n];
  const double d = eps[(size_t)ikp * nb + m] - eps[(size_t)ik * nb + n];
  const double fm = occ[(size_t)ikp * nb + m];
  const double dbar = eps[(size_t)ikp * nb + m] - eps_bar;  // m into an empty state at eps_bar
  for (int iw = 0; iw < nw; ++iw) {
    // kind 0: imaginary-axis frequency i omega_im (+ i eta), real weight;
    // kinds 1 / 2: real part / imaginary part of the complex weight at the
    // real frequency omega_im[iw] with broadening eta
    const int kind = vkind ? vkind[iw] : 0;
    double v = 0.0;
    if (df > occ_tol) {
      double f;
      if (dpole) {
        f = pole_weight(kind, omega_im[iw], eta, dpole[t]);
      } else if (nd > 0) {
        f = 0.0;
        for (int j = 0; j < nd; ++j)
          f += pole_weight(kind, omega_im[iw], eta,
                           epsd[((size_t)ikp * nd + j) * nb + m] - epsd[((size_t)ik * nd + j) * nb + n]);
        f /= nd;
      } else {
        f = pole_weight(kind, omega_im[iw], eta, d);
      }
      v = pref * df * f;
    }
    if (bg && fm > occ_tol) v -= pref * fm * pole_weight(kind, omega_im[iw], eta, dbar);
    w[(size_t)iw * nrow + row] = v;
  }
}

constexpr int kT = 16;     // output tile (complex entries per side)
constexpr int kKB = 32;    // transitions per shared-memory stage
constexpr int kFThreads = 128;
constexpr int kFUnits = 152 * 18;   // blocks: three rounds of six on every SM

__device__ __forceinline__ void tri_decode(int tile, int& I, int& J) {
  int i = (int)((sqrtf(8.0f * (float)tile + 1.0f) - 1.0f) * 0.5f);
  while ((i + 1) * (i + 2) / 2 <= tile) ++i;
  while (i * (i + 1) / 2 > tile) --i;
  I = i;
  J = tile - i * (i + 1) / 2;
}

// part[kc][iw][i][j] = sum_{t in chunk kc} w_t R_ti conj(R_tj) on lower tiles I >= J.
//
// Bound by the FP64 units (2 multiply-adds per clock and SM, 4 per entry and
// transition), so what counts is how few of them are spent beside the lower
// triangle and how evenly the SMs share them: 16 x 16 tiles (N_G = 137: 82% of
// the entries computed are kept, 62% with 32 x 32), the weight multiplied in
// when a row is staged (a thirty-second of the multiply-adds; per use it was a
// fifth), a quadrant of the tile per warp and two entries per lane.  Two stages:
// the rows of one are fetched while the other is summed.  Measured against 32 x
// 32 tiles with four entries per thread: N_G = 137, 5164 rows, 3 frequencies
// 2496 -> 1212 us (1000 us of multiply-adds in the triangle); N_G = 59, 12288 rows
// 338 -> 216 us; N_G = 9, 120 rows 88 -> 6 us (two blocks did all of it).
__global__ void __launch_bounds__(kFThreads, 6)
k_chi0_fp64(const double2* __restrict__ R, const double* __restrict__ w, int64_t nt, int ng,
            int nw, int kchunk, double2* __restrict__ part, const int64_t* __restrict__ perm) {
  __shared__ double2 As[kKB][kT];   // w_t R_ti
  __shared__ double2 Bs[kKB][kT];   // R_tj
  int I, J;
  tri_decode(blockIdx.x, I, J);
  const int kc = blockIdx.y, iw = blockIdx.z;
  const int64_t t0 = (int64_t)kc * kchunk;
  const int64_t t1 = min(nt, t0 + kchunk);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int lr = (warp >> 1) * 8 + (lane >> 2), lc = (warp & 1) * 8 + (lane & 3) * 2;
  const int sc = tid % kT, sr = tid / kT;   // staging: column sc, rows sr, sr + 8, ...
  constexpr int kRows = kKB * kT / kFThreads;
  const int ia = I * kT + sc, ib = J * kT + sc;
  const double* wv = w + (size_t)iw * nt;
  double2 fa[kRows], fb[kRows];
  double fw[kRows];
  auto fetch = [&](int64_t tt) {
#pragma unroll
    for (int q = 0; q < kRows; ++q) {
      const int64_t row = tt + sr + q * (kFThreads / kT);
      fa[q] = fb[q] = make_double2(0.0, 0.0);
      fw[q] = 0.0;
      if (row < t1) {
        const double2* r = R + (perm ? perm[row] : row) * ng;
        if (ia < ng) fa[q] = r[ia];
        if (ib < ng) fb[q] = r[ib];
        fw[q] = wv[row];
      }
    }
  };
  double2 x0 = make_double2(0.0, 0.0), x1 = x0;
  fetch(t0);
  for (int64_t tt = t0; tt < t1; tt += kKB) {
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kRows; ++q) {
      const int r = sr + q * (kFThreads / kT);
      As[r][sc] = make_double2(fw[q] * fa[q].x, fw[q] * fa[q].y);
      Bs[r][sc] = fb[q];
    }
    __syncthreads();
    if (tt + kKB < t1) fetch(tt + kKB);
    const int n = (int)min((int64_t)kKB, t1 - tt);
#pragma unroll 4
    for (int r = 0; r < n; ++r) {
      const double2 a = As[r][lr], b0 = Bs[r][lc], b1 = Bs[r][lc + 1];
      x0.x = fma(a.x, b0.x, x0.x);   // a conj(b)
      x0.y = fma(a.y, b0.x, x0.y);
      x1.x = fma(a.x, b1.x, x1.x);
      x1.y = fma(a.y, b1.x, x1.y);
      x0.x = fma(a.y, b0.y, x0.x);
      x0.y = fma(-a.x, b0.y, x0.y);
      x1.x = fma(a.y, b1.y, x1.x);
      x1.y = fma(-a.x, b1.y, x1.y);
    }
  }
  double2* out = part + ((size_t)kc * nw + iw) * (size_t)ng * ng;
  const int i = I * kT + lr, j = J * kT + lc;
  if (i < ng && j < ng) out[(size_t)i * ng + j] = x0;
  if (i < ng && j + 1 < ng) out[(size_t)i * ng + j + 1] = x1;
}

// chi[iw][i][j] (i >= j) = sum_kc part, then chi[iw][j][i] = conj(chi[iw][i][j]).
// 32 entries of a row per block, their chunks summed by eight warps (a
// thread per entry walked up to hundreds of chunks one load after the other).
constexpr int kRedW = 8;
__global__ void __launch_bounds__(32 * kRedW)
k_chi0_reduce(const double2* __restrict__ part, int nchunks, int ng, int nw, double2* __restrict__ chi,
              int accumulate) {
  __shared__ double2 sums[kRedW][32];
  const int64_t n2 = (int64_t)ng * ng;
  const int iw = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t ij = (int64_t)blockIdx.x * 32 + lane;
  const int i = (int)(ij / ng), j = (int)(ij - (int64_t)i * ng);
  const bool live = ij < n2 && i >= j;
  double2 s = make_double2(0.0, 0.0);
  if (live) {
#pragma unroll 4
    for (int c = warp; c < nchunks; c += kRedW) {
      const double2 v = part[((size_t)c * nw + iw) * n2 + ij];
      s.x += v.x;
      s.y += v.y;
    }
  }
  sums[warp][lane] = s;
  __syncthreads();
  if (warp != 0 || !live) return;
  for (int q = 1; q < kRedW; ++q) {
    s.x += sums[q][lane].x;
    s.y += sums[q][lane].y;
  }
  double2* o = chi + (size_t)iw * n2;
  if (i == j) s.y = 0.0;  // Hermitian: real diagonal
  if (accumulate) {       // add to the sum of the earlier transition blocks
    const double2 a = o[ij];
    s.x += a.x;
    s.y += a.y;
  }
  o[ij] = s;
  if (i != j) o[(size_t)j * ng + i] = make_double2(s.x, -s.y);
}

}  // namespace

cudaError_t launch_weights(int nk, int n_lo, int Nn, int Nm, int nb, const int32_t* kq,
                           const double* eps, const double* occ, const double* omega_im,
                           const int* vkind, int nw, double eta, double pref,
                           double occ_tol, int bg, double eps_bar, const double* dpole, const double* epsd,
                           int nd, double* w, cudaStream_t s, int k0, const int64_t* perm, int64_t nrow) {
  if (!perm) nrow = (int64_t)nk * Nn * Nm;
  if (nrow == 0) return cudaSuccess;
  const int64_t blocks = (nrow + 255) / 256;
  k_weights<<<(unsigned)blocks, 256, 0, s>>>(nk, n_lo, Nn, Nm, nb, kq, eps, occ, omega_im, vkind, nw, eta,
                                            pref, occ_tol, bg, eps_bar, dpole, epsd, nd, w, k0, perm, nrow);
  return cudaGetLastError();
}

int chi0_fp64_chunks(int64_t nt, int ng, int nw) {
  const int64_t nT = (ng + kT - 1) / kT, tiles = nT * (nT + 1) / 2 * nw;
  const int64_t want = (kFUnits + tiles - 1) / tiles;
  const int64_t mem_cap = std::max<int64_t>(1, (int64_t)(8ull << 30) / ((int64_t)ng * ng * nw * 16));
  return (int)std::max<int64_t>(1, std::min({want, mem_cap, (nt + kKB / 2 - 1) / (kKB / 2), (int64_t)65535}));
}

cudaError_t launch_chi0_fp64_partials(const double2* R, const double* w, int64_t nt, int ng,
                                      int nw, int kchunk, int nchunks, double2* part,
                                      cudaStream_t s, const int64_t* perm) {
  const int nT = (ng + kT - 1) / kT;
  dim3 grid((unsigned)(nT * (nT + 1) / 2), (unsigned)nchunks, (unsigned)nw);
  k_chi0_fp64<<<grid, kFThreads, 0, s>>>(R, w, nt, ng, nw, kchunk, part, perm);
  return cudaGetLastError();
}

// chi[iw] = H[v] (imaginary-axis frequency) or H[vr] + i H[vi] (real axis)
__global__ void k_combine_freq(const double2* __restrict__ H, const int* __restrict__ vr,
                               const int* __restrict__ vi, int64_t n2, double2* __restrict__ chi) {
  const int iw = blockIdx.y;
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n2) return;
  const double2 a = H[(size_t)vr[iw] * n2 + e];
  double2 v = a;
  if (vi[iw] >= 0) {
    const double2 b = H[(size_t)vi[iw] * n2 + e];
    v = make_double2(a.x - b.y, a.y + b.x);
  }
  chi[(size_t)iw * n2 + e] = v;
}

cudaError_t launch_combine_freq(const double2* H, const int* vr, const int* vi, int ng, int nw, double2* chi,
                                cudaStream_t s) {
  const int64_t n2 = (int64_t)ng * ng;
  k_combine_freq<<<dim3((unsigned)((n2 + 255) / 256), (unsigned)nw), 256, 0, s>>>(H, vr, vi, n2, chi);
  return cudaGetLastError();
}

cudaError_t launch_chi0_reduce(const double2* part, int nchunks, int ng, int nw, double2* chi,
                               cudaStream_t s, int accumulate) {
  const dim3 grid((unsigned)(((int64_t)ng * ng + 31) / 32), (unsigned)nw);
  k_chi0_reduce<<<grid, 32 * kRedW, 0, s>>>(part, nchunks, ng, nw, chi, accumulate);
  return cudaGetLastError();
}

}  // namespace chi0
