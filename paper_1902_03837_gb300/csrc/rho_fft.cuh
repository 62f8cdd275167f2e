// Oscillator strengths through in-register transforms on a small alias-free
// grid (kernels; instantiated per type in rho_fft32.cu / rho_fft64.cu).
//
//   rho(G) = 1/N^3 sum_r conj(u_n(r)) u_m(r) e^{i h.r},   h = G - G0,
//
// is exact on every grid with N > 2 L + max|h| per axis (L: largest Miller
// index of the spheres, over both signs and every k), so the states are put on
// the smallest such N^3 grid that the column transform (fft.cuh) knows, whatever
// grid the caller set.  The bound is sufficient, not necessary: spheres and response
// sets that lie off-centre can be alias free with a few points less.
// For the 48^3 grid of the precision workload that is 24^3: an eighth of the
// points.  The result is the same sum; only its rounding differs.
//
// Measured against the mixed-grid kernels of rho.cu on the caller's grid
// (states and rho together, one GB300): 6x6x6 k, 16 + 184 bands, N_G = 1000,
// 48^3 -> 24^3, FP32: 181 -> 20.2 ms; 4x4x4 k, 64 bands, N_G = 431, 30^3 ->
// 20^3, FP32: 13.7 -> 1.5 ms; 4x4x4 k, 8 + 24 bands, N_G = 59, 24^3 -> 12^3,
// FP64: 12.3 -> 0.85 ms.
//
// Per transition the three axes are transformed one after the other and cut
// to the response set after each: z columns straight from the two states'
// real-space columns (product in registers), y columns of the HZ planes kept,
// x columns of the (y, z) pairs that hold response vectors.  Between the axes
// the data goes through shared memory once: N HZ values per x plane, and
// N values per pair.  One thread transforms one column, so a column costs no
// barriers, and 5 N log2 N additions in place of N HZ multiply-adds.
#pragma once

#include "fft.cuh"
#include "internal.cuh"

namespace chi0 {

namespace rfft {

constexpr int kMaxThreads = 256;
// Blocks that the registers of rho's kernel leave room for on an SM.
template <typename T, int N>
constexpr int kRhoBlocks = sizeof(T) == 4 || N <= 16 ? 2 : 1;

// frequency of output (and input) i of an N-point column, in [-N/2, N/2)
template <int N, int I>
constexpr int kFreq = I < (N + 1) / 2 ? I : I - N;

// ---------------------------------------------------------------------------
// States: c(G) on the k sphere -> u(x, z, y) = sum_G c(G) e^{2 pi i G.r / N},
// one block per (k, band).  x columns in place in the box of the sphere
// (N x NY x NZ), then y and z columns of xc planes at a time; z columns go to
// HBM with y fastest, so every access of a warp is contiguous.
// ---------------------------------------------------------------------------
template <typename T, int N>
__global__ void __launch_bounds__(kMaxThreads, sizeof(T) == 4 ? 2 : 1)
k_wf_fft(RhoGeom g, const int32_t* __restrict__ gvec, const int32_t* __restrict__ npw,
         const typename C2<T>::t* __restrict__ coef, typename C2<T>::t* __restrict__ U, int k0, int b0, int nbo,
         int xc) {
  using T2 = typename C2<T>::t;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int NY = g.NY, NZ = g.NZ, nyz = NY * NZ;
  T2* box = reinterpret_cast<T2*>(smem_raw);  // [N][NY][NZ]
  T2* mid = box + (size_t)N * nyz;            // [xc][N][NZ]
  const int tid = threadIdx.x, nth = blockDim.x;
  const int ikl = blockIdx.x / nbo, bl = blockIdx.x - ikl * nbo;
  const int ik = k0 + ikl, band = b0 + bl;
  T2 zero;
  zero.x = 0;
  zero.y = 0;
  for (int i = tid; i < N * nyz; i += nth) box[i] = zero;
  __syncthreads();
  {
    const int np = npw[ik];
    const int32_t* gv = gvec + (size_t)ik * g.npw_max * 3;
    const T2* c = coef + ((size_t)ik * g.nb + band) * g.npw_max;
    for (int p = tid; p < np; p += nth) {
      const int gx = gv[3 * p], gy = gv[3 * p + 1], gz = gv[3 * p + 2];
      box[((gx < 0 ? gx + N : gx) * NY + gy + g.Ly) * NZ + gz + g.Lz] = c[p];
    }
  }
  __syncthreads();
  for (int u = tid; u < nyz; u += nth) {
    T2 a[N];
    T2* col = box + u;
    fft::static_for<0, N>([&](auto ic) { a[ic.value] = col[ic.value * nyz]; });
    fft::column<N>(a);
    fft::static_for<0, N>([&](auto ic) { col[ic.value * nyz] = a[ic.value]; });
  }
  __syncthreads();
  T2* out = U + ((size_t)ikl * nbo + bl) * (size_t)(N * N * N);
  for (int x0 = 0; x0 < N; x0 += xc) {
    const int nx = min(xc, N - x0);
    for (int u = tid; u < nx * NZ; u += nth) {
      const int xl = u / NZ, gz = u - xl * NZ;
      T2 a[N];
      const T2* col = box + ((size_t)(x0 + xl) * NY + g.Ly) * NZ + gz;
      fft::static_for<0, N>([&](auto ic) {
        constexpr int i = decltype(ic)::value, h = kFreq<N, i>;
        a[i] = (h < 0 ? -h : h) <= g.Ly ? col[h * NZ] : zero;
      });
      fft::column<N>(a);
      T2* o = mid + (size_t)xl * N * NZ + gz;
      fft::static_for<0, N>([&](auto ic) { o[ic.value * NZ] = a[ic.value]; });
    }
    __syncthreads();
    for (int u = tid; u < nx * N; u += nth) {
      const int xl = u / N, y = u - xl * N;
      T2 a[N];
      const T2* col = mid + (size_t)u * NZ + g.Lz;
      fft::static_for<0, N>([&](auto ic) {
        constexpr int i = decltype(ic)::value, h = kFreq<N, i>;
        a[i] = (h < 0 ? -h : h) <= g.Lz ? col[h] : zero;
      });
      fft::column<N>(a);
      T2* o = out + (size_t)(x0 + xl) * (N * N) + y;
      fft::static_for<0, N>([&](auto ic) { o[ic.value * N] = a[ic.value]; });
    }
    __syncthreads();
  }
}

// conj(a) b
template <typename T2>
__device__ __forceinline__ T2 cjmul(const T2 a, const T2 b) {
  T2 r;
  r.x = fma(a.x, b.x, a.y * b.y);
  r.y = fma(a.x, b.y, -a.y * b.x);
  return r;
}

// ---------------------------------------------------------------------------
// rho of one n at k and up to jm consecutive m at k - q (the same block order
// and output as the generic kernel of rho.cu).
//
// Bound by the FP32 (FP64) pipes.  In FP32 the n column stays in registers over
// the block's m bands while both fit (kResident); the states are read from L2
// once per block (1 + 1/jm volumes per transition).  In FP64 the registers are
// worth more as resident warps, and the columns of all m bands are dealt out
// one by one, so that fewer lanes idle in the last warp (12^3, 12288
// transitions: 900 -> 695 us, of which the FP64 operations take 600).  zs is padded to an odd row so
// that the y columns of a warp (stride N | 1) fall into distinct banks.
// ---------------------------------------------------------------------------
template <typename T, int N>
__device__ __forceinline__ void rho_fft_block(const RhoTask<T, typename C2<T>::t>& tk, int64_t blk,
                                              unsigned char* smem_raw) {
  using T2 = typename C2<T>::t;
  constexpr int NP = N | 1;
  constexpr bool kResident = sizeof(T) == 4 && N <= 24;
  const RhoGeom& g = tk.g;
  const int tid = threadIdx.x, nth = blockDim.x;
  const int jm = tk.jm, xc = tk.xc, P = g.npair, HZ = g.HZ, HX = g.HX;
  const int nmc = (g.Nm + jm - 1) / jm;
  const int mc = (int)(blk % nmc);
  const int nrel = (int)((blk / nmc) % g.Nn);
  const int ik = (int)(blk / ((int64_t)nmc * g.Nn));
  const int m0 = mc * jm;
  const int cm = min(jm, g.Nm - m0);
  const int ikg = g.k0 + ik;
  const int ikp = tk.kq[ikg];
  const int hx_base = g.Mx_lo - tk.g0[3 * ikg];
  const int hy_base = g.My_lo - tk.g0[3 * ikg + 1];
  const int hz_base = g.Mz_lo - tk.g0[3 * ikg + 2];
  const size_t vol = (size_t)N * N * N;
  const int nbu = g.nbu ? g.nbu : g.nb, nbm = g.nbm ? g.nbm : g.nb;
  const T2* __restrict__ Un = tk.U + ((size_t)ik * nbu + (g.n_lo - g.bu0 + nrel)) * vol;
  const T2* __restrict__ Um =
      (tk.Um ? tk.Um : tk.U) + ((size_t)ikp * nbm + m0 + (g.diag ? g.n_lo + nrel : 0)) * vol;

  T2* xb = reinterpret_cast<T2*>(smem_raw);     // [cm][N][P]
  T2* zs = xb + (size_t)jm * N * P;             // [cm][nx][HZ][NP]; the output rows [cm][ng] after the last plane

  for (int x0 = 0; x0 < N; x0 += xc) {
    const int nx = min(xc, N - x0);
    // z columns of the products: zs[j][xl][hz][y]
    auto store = [&](const T2 (&a)[N], T2* o) {
      fft::static_for<0, N>([&](auto ic) {
        constexpr int i = decltype(ic)::value, h = kFreq<N, i>;
        if ((unsigned)(h - hz_base) < (unsigned)HZ) o[h * NP] = a[i];
      });
    };
    if constexpr (kResident) {
      for (int u = tid; u < nx * N; u += nth) {
        const int xl = u / N, y = u - xl * N;
        const size_t off = (size_t)(x0 + xl) * (N * N) + y;
        T2 un[N];
        fft::static_for<0, N>([&](auto ic) { un[ic.value] = __ldg(Un + off + ic.value * N); });
        T2* o = zs + ((size_t)xl * HZ - hz_base) * NP + y;
        for (int j = 0; j < cm; ++j) {
          const T2* __restrict__ um = Um + (size_t)j * vol + off;
          T2 a[N];
          fft::static_for<0, N>([&](auto ic) { a[ic.value] = __ldg(um + ic.value * N); });
          fft::static_for<0, N>([&](auto ic) { a[ic.value] = cjmul(un[ic.value], a[ic.value]); });
          fft::column<N>(a);
          store(a, o);
          o += (size_t)nx * HZ * NP;
        }
      }
    } else {
      for (int u = tid; u < cm * nx * N; u += nth) {
        const int r = u / N, y = u - r * N;   // r = j nx + xl
        const int j = r / nx;
        const size_t off = (size_t)(x0 + r - j * nx) * (N * N) + y;
        const T2* __restrict__ um = Um + (size_t)j * vol + off;
        T2 a[N];
        fft::static_for<0, N>([&](auto ic) { a[ic.value] = __ldg(um + ic.value * N); });
        fft::static_for<0, N>([&](auto ic) { a[ic.value] = cjmul(__ldg(Un + off + ic.value * N), a[ic.value]); });
        fft::column<N>(a);
        store(a, zs + ((size_t)r * HZ - hz_base) * NP + y);
      }
    }
    __syncthreads();
    // y columns: xb[j][x][pair]
    for (int u = tid; u < cm * nx * HZ; u += nth) {
      const int r = u / HZ, hz = u - r * HZ;
      const int j = r / nx, xl = r - j * nx;
      T2 a[N];
      const T2* col = zs + (size_t)u * NP;
      fft::static_for<0, N>([&](auto ic) { a[ic.value] = col[ic.value]; });
      fft::column<N>(a);
      const int32_t row = __ldg(g.rows + hz);   // first pair | first hy | number of hy
      const int lo = hy_base + ((row >> 8) & 0xff), cnt = row & 0xff;
      T2* o = xb + (size_t)(j * N + x0 + xl) * P + (row >> 16) - lo;
      fft::static_for<0, N>([&](auto ic) {
        constexpr int i = decltype(ic)::value, h = kFreq<N, i>;
        if ((unsigned)(h - lo) < (unsigned)cnt) o[h] = a[i];
      });
    }
    __syncthreads();
  }
  // x columns of the pairs, put in the order of the response set in zs.  1 / N^3
  // in FP32 carries its rounding error along: rounded alone it would shift every
  // rho by the same 3e-8 and chi0 by twice that, which no sum averages out.
  constexpr double inv = 1.0 / ((double)N * N * N);
  constexpr T scale = (T)inv;
  auto scaled = [&](T v) {
    if constexpr (sizeof(T) == 4) {
      constexpr T rest = (T)(inv - (double)scale);
      return fma(v, scale, v * rest);
    } else {
      return v * scale;
    }
  };
  for (int u = tid; u < cm * P; u += nth) {
    const int j = u / P, p = u - j * P;
    T2 a[N];
    const T2* col = xb + (size_t)j * N * P + p;
    fft::static_for<0, N>([&](auto ic) { a[ic.value] = col[ic.value * P]; });
    fft::column<N>(a);
    T2* o = zs + (size_t)j * g.ng;
    const int16_t* lut = g.lut + p - hx_base * P;
    fft::static_for<0, N>([&](auto ic) {
      constexpr int i = decltype(ic)::value, h = kFreq<N, i>;
      if ((unsigned)(h - hx_base) < (unsigned)HX) {
        const int k = __ldg(lut + h * P);
        if (k >= 0) {
          a[i].x = scaled(a[i].x);
          a[i].y = scaled(a[i].y);
          o[k] = a[i];
        }
      }
    });
  }
  __syncthreads();
  T2* R = tk.R + (((int64_t)ik * g.Nn + nrel) * g.Nm + m0) * g.ng;
  for (int i = tid; i < cm * g.ng; i += nth) R[i] = zs[i];
}

template <typename T, int N>
__global__ void __launch_bounds__(kMaxThreads, kRhoBlocks<T, N>)
k_rho_fft(const RhoTask<T, typename C2<T>::t> tk) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  rho_fft_block<T, N>(tk, blockIdx.x, smem_raw);
}

// Persistent form over the tasks of one grid size (as k_rho_batch of rho.cu).
template <typename T, int N>
__global__ void __launch_bounds__(kMaxThreads, kRhoBlocks<T, N>)
k_rho_fft_batch(const RhoTask<T, typename C2<T>::t>* __restrict__ tasks, int ntasks, int64_t total,
                unsigned long long* __restrict__ counter) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ RhoTask<T, typename C2<T>::t> stk;
  __shared__ long long snext;
  for (;;) {
    if (threadIdx.x == 0) {
      snext = (long long)atomicAdd(counter, 1ull);
      if (snext < total) {
        int lo = 0, hi = ntasks - 1;  // last task with block0 <= snext
        while (lo < hi) {
          const int mid = (lo + hi + 1) / 2;
          if (tasks[mid].block0 <= snext) lo = mid; else hi = mid - 1;
        }
        stk = tasks[lo];
      }
    }
    __syncthreads();
    if (snext >= total) break;
    rho_fft_block<T, N>(stk, snext - stk.block0, smem_raw);
    __syncthreads();
  }
}

// ---- host side ----

template <typename T, int N>
cudaError_t wf_launch(const RhoGeom& g, const int32_t* gvec, const int32_t* npw, const typename C2<T>::t* coef,
                      typename C2<T>::t* U, cudaStream_t s, int k0, int nkr, int b0, int nbo) {
  using T2 = typename C2<T>::t;
  const size_t box = (size_t)N * g.NY * g.NZ * sizeof(T2), per = (size_t)N * g.NZ * sizeof(T2);
  // planes per pass: as many as leave room for three blocks on an SM, else two
  int xc = 1;
  for (size_t lim : {(size_t)74 << 10, (size_t)112 << 10, (size_t)227 << 10})
    if (box + 2 * per <= lim) {
      xc = (int)((lim - box) / per);
      if (xc > N) xc = N;
      break;
    }
  xc = (N + (N + xc - 1) / xc - 1) / ((N + xc - 1) / xc);   // passes of equal size
  const size_t smem = box + xc * per;
  if (smem > (227 << 10)) return cudaErrorInvalidValue;
  cudaError_t e =
      cudaFuncSetAttribute(k_wf_fft<T, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_limit());
  if (e != cudaSuccess) return e;
  k_wf_fft<T, N><<<nkr * nbo, kMaxThreads, smem, s>>>(g, gvec, npw, coef, U, k0, b0, nbo, xc);
  return cudaGetLastError();
}

template <typename T, int N>
cudaError_t rho_launch(const RhoTask<T, typename C2<T>::t>& tk, size_t smem, int threads, int64_t nblocks,
                       cudaStream_t s) {
  cudaError_t e =
      cudaFuncSetAttribute(k_rho_fft<T, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_limit());
  if (e != cudaSuccess) return e;
  k_rho_fft<T, N><<<(unsigned)nblocks, threads, smem, s>>>(tk);
  return cudaGetLastError();
}

template <typename T, int N>
cudaError_t batch_launch(const RhoTask<T, typename C2<T>::t>* tasks, int ntasks, int64_t total, size_t smem,
                         unsigned long long* counter, int grid, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(k_rho_fft_batch<T, N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       smem_limit(sizeof(RhoTask<T, typename C2<T>::t>) + 8));
  if (e != cudaSuccess) return e;
  k_rho_fft_batch<T, N><<<(unsigned)(total < grid ? total : grid), kMaxThreads, smem, s>>>(tasks, ntasks, total, counter);
  return cudaGetLastError();
}

// calls F<N> for the size n (a size of kRhoFftSizes)
#define CHI0_RHO_FFT_SWITCH(n, CALL)         \
  switch (n) {                               \
    case 8: return CALL(8);                  \
    case 10: return CALL(10);                \
    case 12: return CALL(12);                \
    case 15: return CALL(15);                \
    case 16: return CALL(16);                \
    case 18: return CALL(18);                \
    case 20: return CALL(20);                \
    case 24: return CALL(24);                \
    case 30: return CALL(30);                \
    case 32: return CALL(32);                \
    case 36: return CALL(36);                \
    default: return cudaErrorInvalidValue;   \
  }

template <typename T>
cudaError_t wf_dispatch(const RhoGeom& g, const int32_t* gvec, const int32_t* npw, const typename C2<T>::t* coef,
                        typename C2<T>::t* U, cudaStream_t s, int k0, int nkr, int b0, int nbo) {
#define CHI0_CALL(n) wf_launch<T, n>(g, gvec, npw, coef, U, s, k0, nkr, b0, nbo)
  CHI0_RHO_FFT_SWITCH(g.nfft, CHI0_CALL)
#undef CHI0_CALL
}
template <typename T>
cudaError_t rho_dispatch(const RhoTask<T, typename C2<T>::t>& tk, size_t smem, int threads, int64_t nblocks,
                         cudaStream_t s) {
#define CHI0_CALL(n) rho_launch<T, n>(tk, smem, threads, nblocks, s)
  CHI0_RHO_FFT_SWITCH(tk.g.nfft, CHI0_CALL)
#undef CHI0_CALL
}
template <typename T>
cudaError_t batch_dispatch(int nfft, const RhoTask<T, typename C2<T>::t>* tasks, int ntasks, int64_t total,
                           size_t smem, unsigned long long* counter, int grid, cudaStream_t s) {
#define CHI0_CALL(n) batch_launch<T, n>(tasks, ntasks, total, smem, counter, grid, s)
  CHI0_RHO_FFT_SWITCH(nfft, CHI0_CALL)
#undef CHI0_CALL
}

}  // namespace rfft

}  // namespace chi0
