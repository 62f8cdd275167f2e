// Self-energy kernel I of the full-frequency GW step (Eqs. W_def, W_delta, I_c):
//
//   I^{ab k}_{m q}(w) = -1/(N_k Omega) sum_{G,G'} W^d_GG'(q,w) rho_{amk}(q,G) conj(rho_{bmk}(q,G')),
//
// W = V eps~^-1 V (the symmetric form of Eq. W_def), W^d its delta-like part
// (Eq. W_delta), a and b two bands of the quasiparticle window at k, m any
// band at k - q.  With Y(i, t) = sum_j W^d_ij conj(rho_t(j)) (the contraction:
// tensor cores in the mixed form, tc.cu; the plain FP64 kernel below in the
// FP64 form) every entry is one dot product over i:
//
//   I[k][m][a][b] = -1/(N_k Omega) sum_i rho_{(k,m,a)}(i) Y(i, (k,m,b)).
//
// Transitions of the window are ordered t = ((k nb) + m) nqp + a (partners of
// one (k, m) adjacent); the rho kernel writes them in the order
// ((k nqp) + a) nb + m.  Y is stored as 64 x 64 complex tiles, tile
// (i / 64) + (t / 64) * nI, nI = ceil(ng / 64), entry (i % 64) * 64 + t % 64,
// in FP32 (mixed form) or FP64; rho is copied once per call into the same
// layout (RT) for the dot products.
#include "internal.cuh"

namespace chi0 {

namespace {

__device__ __forceinline__ int64_t rho_row(int64_t t, int nqp, int nb) {
  const int64_t a = t % nqp, g = t / nqp;
  return ((g / nb) * nqp + a) * nb + g % nb;
}

// W^d_ij = V_i V_j [ (Im E_ij + Im E_ji) / 2 - i (Re E_ij - Re E_ji) / 2 ] in FP64
__global__ void k_sig_wd64(const double2* __restrict__ E, const double* __restrict__ v, int ng,
                           double2* __restrict__ Wd) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)ng * ng) return;
  const int i = (int)(e / ng), j = (int)(e % ng);
  const double2 a = E[e], b = E[(size_t)j * ng + i];
  const double f = 0.5 * v[i] * v[j];
  Wd[e] = make_double2(f * (a.y + b.y), -f * (a.x - b.x));
}

// Y(i, t) = sum_j W^d_ij conj(rho_t(j)), plain FP64: 16 x 16 outputs per
// block, 16-wide slices of j staged in shared memory.  Bound by the FP64 units:
// four multiply-adds per product (six operations when written as
// sums of products: N_G = 123, 9912 columns, 8 frequencies 17.5 ms, 11.3 so).
__global__ void __launch_bounds__(256)
k_sig_gemm64(const double2* __restrict__ Wd, const double2* __restrict__ R, int ng, int64_t T, int nqp, int nb,
             int nI, double2* __restrict__ Y) {
  __shared__ double2 ws[16][17], rs[16][17];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int i0 = blockIdx.y * 16;
  const int64_t t0 = (int64_t)blockIdx.x * 16;
  const int i = i0 + ty;
  const int64_t t = t0 + tx;
  const int64_t lrow = (t0 + ty < T) ? rho_row(t0 + ty, nqp, nb) : -1;   // the row this thread stages
  double sx = 0.0, sy = 0.0;
  for (int j0 = 0; j0 < ng; j0 += 16) {
    const int j = j0 + tx;
    ws[ty][tx] = (i0 + ty < ng && j < ng) ? Wd[(size_t)(i0 + ty) * ng + j] : make_double2(0.0, 0.0);
    const double2 r = (lrow >= 0 && j < ng) ? R[lrow * ng + j] : make_double2(0.0, 0.0);
    rs[ty][tx] = make_double2(r.x, -r.y);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const double2 a = ws[ty][q], b = rs[tx][q];
      sx = fma(a.x, b.x, sx);
      sx = fma(-a.y, b.y, sx);
      sy = fma(a.x, b.y, sy);
      sy = fma(a.y, b.x, sy);
    }
    __syncthreads();
  }
  if (i < ng && t < T)
    Y[((size_t)(t / 64) * nI + i / 64) * 4096 + (size_t)(i % 64) * 64 + t % 64] = make_double2(sx, sy);
}

constexpr int kDotUnroll = 4;   // values of i per thread between compensated sums

__device__ __forceinline__ size_t tile_off(int64_t t, int i, int nI) {
  return ((size_t)(t >> 6) * nI + (i >> 6)) * 4096 + (size_t)(i & 63) * 64 + (t & 63);
}

// rho of the window in the tile layout of Y: RT(i, t) = rho_t(i), t in the
// group-major order (one pass per call; the dot then reads its columns
// coalesced).  32 x 32 blocks through shared memory.
template <typename TR>
__global__ void __launch_bounds__(256)
k_sig_rhot(const TR* __restrict__ R, int64_t T, int nqp, int nb, int ng, int nI, TR* __restrict__ RT) {
  __shared__ TR tl[32][33];
  const int64_t t0 = (int64_t)blockIdx.x * 32;
  const int i0 = blockIdx.y * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // 8 rows per pass
  for (int r = ty; r < 32; r += 8) {
    const int64_t t = t0 + r;
    const int i = i0 + tx;
    TR v;
    v.x = 0;
    v.y = 0;
    if (t < T && i < ng) v = R[rho_row(t, nqp, nb) * ng + i];
    tl[r][tx] = v;
  }
  __syncthreads();
  for (int r = ty; r < 32; r += 8) {
    const int i = i0 + r;
    const int64_t t = t0 + tx;
    if (t < T && i < ng) RT[tile_off(t, i, nI)] = tl[tx][r];
  }
}

// Running sum of the dot products: FP64 in the FP64 form; in the mixed form
// FP32 with Neumaier compensation (GB300's FP64 units are too few to convert
// and add every partial sum in FP64 at the rate the loads arrive).
template <typename F>
struct DotSum {
  F s = 0, c = 0;
  __device__ __forceinline__ void add(F x) {
    if constexpr (sizeof(F) == 4) {
      const F t = s + x;
      c += (fabsf(s) >= fabsf(x)) ? ((s - t) + x) : ((x - t) + s);
      s = t;
    } else {
      s += x;
    }
  }
  __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};

// I[g][a][b] = pref sum_i rho_{(g,a)}(i) Y(i, (g,b)), g = (k, m): one block
// per 32 columns t = (g, b) and frequency; 256 threads = 32 columns x 8 phases
// over i (64 columns x 4 phases left 1.7 blocks per SM at 16384 columns, each
// thread walking twice as far: 34 -> 28 us per frequency of N_G = 300).
// Each thread reads its column of Y and the columns (g, a) of RT (tile
// layout, both coalesced across the warp), A partners per pass.  Products in
// the element type of rho, summed kDotUnroll at a time into a DotSum.
// Bound by the latency of its loads (the data comes mostly from L2): all of a
// step's loads are issued together, the last ragged step's as well (its rows
// repeat the last one, with Y as 0), and with kQuad (FP32, a multiple of A
// partners, so that a group's columns start on 16 bytes) two partners come per
// load: N_G = 300, 16384 columns, two frequencies 55 -> 46 us.
constexpr int kDotP = 8;
template <typename TR, typename TY, int A, bool kQuad>
__global__ void __launch_bounds__(32 * kDotP, (sizeof(TR) == 8 && A == 4) ? 3 : 1)
k_sig_dot(const TR* __restrict__ RT, const TY* __restrict__ Y, int ng, int64_t T, int nqp, int nI, double pref,
          double2* __restrict__ out, size_t ystride, size_t ostride) {
  using F = decltype(TR::x);
  __shared__ double2 red[kDotP][32][A];
  Y += blockIdx.y * ystride;
  out += blockIdx.y * ostride;
  const int jl = threadIdx.x & 31, ph = threadIdx.x >> 5;
  const int64_t t = (int64_t)blockIdx.x * 32 + jl;
  const bool live = t < T;
  const int64_t g = live ? t / nqp : 0;
  const int b = live ? (int)(t % nqp) : 0;
  const TY* Ycol = Y + tile_off(t, 0, nI);
  for (int a0 = 0; a0 < nqp; a0 += A) {
    const TR* col[A];   // the partners (g, a0 + q) in RT
#pragma unroll
    for (int q = 0; q < A; ++q) col[q] = RT + tile_off(g * nqp + ((a0 + q < nqp) ? a0 + q : 0), 0, nI);
    DotSum<F> sx[A], sy[A];
    if (live) {
      for (int i0 = ph; i0 < ng; i0 += kDotP * kDotUnroll) {
        TY yv[kDotUnroll];
        TR rv[kDotUnroll][A];
#pragma unroll
        for (int r = 0; r < kDotUnroll; ++r) {
          const int i = i0 + kDotP * r, ic = i < ng ? i : ng - 1;
          const size_t ro = (size_t)(ic >> 6) * 4096 + (size_t)(ic & 63) * 64;
          yv[r] = Ycol[ro];
          if (i >= ng) yv[r].x = yv[r].y = 0;
          if constexpr (kQuad) {
#pragma unroll
            for (int q = 0; q < A; q += 2) {
              const float4 v = *reinterpret_cast<const float4*>(col[q] + ro);
              rv[r][q].x = v.x;
              rv[r][q].y = v.y;
              rv[r][q + 1].x = v.z;
              rv[r][q + 1].y = v.w;
            }
          } else {
#pragma unroll
            for (int q = 0; q < A; ++q) rv[r][q] = col[q][ro];
          }
        }
        F cx[A], cy[A];
#pragma unroll
        for (int q = 0; q < A; ++q) cx[q] = cy[q] = 0;
#pragma unroll
        for (int r = 0; r < kDotUnroll; ++r) {
          const F yx = (F)yv[r].x, yy = (F)yv[r].y;
#pragma unroll
          for (int q = 0; q < A; ++q) {   // (partners past nqp repeat one that is not written)
            cx[q] = fma(rv[r][q].x, yx, cx[q]);
            cx[q] = fma(-rv[r][q].y, yy, cx[q]);
            cy[q] = fma(rv[r][q].x, yy, cy[q]);
            cy[q] = fma(rv[r][q].y, yx, cy[q]);
          }
        }
#pragma unroll
        for (int q = 0; q < A; ++q) {
          sx[q].add(cx[q]);
          sy[q].add(cy[q]);
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < A; ++q) red[ph][jl][q] = make_double2(sx[q].value(), sy[q].value());
    __syncthreads();
    // thread (ph, jl) adds the phases of partner a0 + ph
    if (live && ph < A && a0 + ph < nqp) {
      double x = 0.0, y = 0.0;
#pragma unroll
      for (int p = 0; p < kDotP; ++p) {
        x += red[p][jl][ph].x;
        y += red[p][jl][ph].y;
      }
      out[((size_t)g * nqp + a0 + ph) * nqp + b] = make_double2(pref * x, pref * y);
    }
  }
}
static_assert(kDotP >= 8, "one phase per partner of a pass");

}  // namespace

cudaError_t launch_sig_wd64(const double2* E, const double* vsqrt, int ng, double2* Wd, cudaStream_t s) {
  const int64_t n = (int64_t)ng * ng;
  k_sig_wd64<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(E, vsqrt, ng, Wd);
  return cudaGetLastError();
}

cudaError_t launch_sig_gemm64(const double2* Wd, const double2* R, int ng, int64_t T, int nqp, int nb,
                              double2* Y, cudaStream_t s) {
  const int nI = (ng + 63) / 64;
  k_sig_gemm64<<<dim3((unsigned)((T + 15) / 16), (unsigned)((ng + 15) / 16)), 256, 0, s>>>(Wd, R, ng, T, nqp,
                                                                                          nb, nI, Y);
  return cudaGetLastError();
}

template <typename TR>
cudaError_t launch_sig_rhot(const TR* R, int64_t T, int nqp, int nb, int ng, TR* RT, cudaStream_t s) {
  const int nI = (ng + 63) / 64;
  k_sig_rhot<TR><<<dim3((unsigned)((T + 31) / 32), (unsigned)((ng + 31) / 32)), 256, 0, s>>>(R, T, nqp, nb, ng, nI,
                                                                                              RT);
  return cudaGetLastError();
}

template <typename TR, typename TY>
cudaError_t launch_sig_dot(const TR* RT, const TY* Y, int ng, int64_t T, int nqp, double pref, double2* out,
                           cudaStream_t s, int nf, size_t ystride, size_t ostride) {
  const int nI = (ng + 63) / 64;
  const dim3 grid((unsigned)((T + 31) / 32), (unsigned)nf);
  constexpr bool f32 = sizeof(TR) == 8;
  // up to 4 partners per pass: fewer registers, more resident blocks
  auto kernel = nqp <= 4 ? (f32 && nqp == 4 ? k_sig_dot<TR, TY, 4, f32> : k_sig_dot<TR, TY, 4, false>)
                         : (f32 && nqp % 8 == 0 ? k_sig_dot<TR, TY, 8, f32> : k_sig_dot<TR, TY, 8, false>);
  kernel<<<grid, 32 * kDotP, 0, s>>>(RT, Y, ng, T, nqp, nI, pref, out, ystride, ostride);
  return cudaGetLastError();
}

template cudaError_t launch_sig_rhot<float2>(const float2*, int64_t, int, int, int, float2*, cudaStream_t);
template cudaError_t launch_sig_rhot<double2>(const double2*, int64_t, int, int, int, double2*, cudaStream_t);
template cudaError_t launch_sig_dot<float2, float2>(const float2*, const float2*, int, int64_t, int, double,
                                                    double2*, cudaStream_t, int, size_t, size_t);
template cudaError_t launch_sig_dot<double2, double2>(const double2*, const double2*, int, int64_t, int, double,
                                                      double2*, cudaStream_t, int, size_t, size_t);

}  // namespace chi0
