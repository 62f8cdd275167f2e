// Dyson step of the Linear Algebra subsection (Eqs. X_rpa, X_rpa_inv) in the
// symmetric form used for W (Eq. W_def):
//
//     eps~ = 1 - V chi0 V,   V = diag(sqrt(4 pi) / |q+G|),   out = eps~^-1,
//
// one matrix per frequency, all frequencies of a group in one batch.  On the
// imaginary axis eps~ is Hermitian positive definite (chi0 is negative
// semidefinite), so the inverse is taken by blocked in-place Gauss-Jordan
// elimination without pivoting.  For the pivot block b (16 columns), with
// P = A_bb^-1:
//
//     A_ij <- A_ij - A_ib P A_bj     (i, j outside b)
//     A_bj <- P A_bj,   A_ib <- -A_ib P,   A_bb <- P,
//
// and after the last block A holds eps~^-1.  FP64 throughout.
//
// Symmetry halves the work: once the rows/columns of a set S have been swept,
// A_ji = s conj(A_ij) with s = -1 when exactly one of i, j lies in S and +1
// otherwise.  Only the tiles on and below the diagonal are updated; the
// panels read entries above the diagonal through that rule, and the last step
// writes the conjugates of the lower tiles into the upper ones.
//
// What bounds it: the FP64 units, 2 multiply-adds per clock and SM (2 N_G^3
// of them per matrix), and for small matrices or few of them the chain
// pivot -> panels -> update.  At that rate a 32 x 32 complex block takes an SM
// 34 us to multiply and as long to invert, so blocks of 16 and a split of the
// chain over SMs decide: the pivot of block b + 1 is updated and inverted by a
// block of its own (one SM) while the others still update with block b, eps~
// is formed from chi0 where the first step reads it, and the mirror pass is
// part of the last step, which leaves two launches per 16 columns.  Measured
// against blocks of 32 with a pivot kernel of its own (about 140 us each) and
// separate passes for eps~ and the mirror: 12 matrices of N_G = 300 21.5 ->
// 1.70 ms (all at a time instead of one by one; the multiply-adds alone take
// 1.1 ms), one of N_G = 59 0.32 -> 0.14 ms.
#include "internal.cuh"

namespace chi0 {

namespace {

constexpr int kNB = 16;         // pivot block width and tile edge
constexpr int kThreads = 128;   // 4 warps, one tile each
constexpr int kPE = 8;          // columns per block of the panels

// complex arithmetic as fused multiply-adds (4 per multiply-add): the FP64
// units are the bound of this step
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ void cmac(double2& acc, double2 a, double2 b) {  // acc += a b
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(a.y, b.x, acc.y);
}
__device__ __forceinline__ void cmsub(double2& acc, double2 a, double2 b) {  // acc -= a b
  acc.x = fma(-a.x, b.x, acc.x);
  acc.x = fma(a.y, b.y, acc.x);
  acc.y = fma(-a.x, b.y, acc.y);
  acc.y = fma(-a.y, b.x, acc.y);
}

// The matrices of one call, and element (i, j) of eps~ as a step reads it:
// from chi0 in the first step, from A afterwards.
struct Mats {
  const double2* chi;
  const double* v;
  double2* A;
  int ng;
  __device__ __forceinline__ double2 get(int iw, int i, int j, bool first) const {
    const size_t e = (size_t)iw * ng * ng + (size_t)i * ng + j;
    if (!first) return A[e];
    const double s = -__ldg(v + i) * __ldg(v + j);
    const double2 c = chi[e];
    return make_double2((i == j ? 1.0 : 0.0) + s * c.x, s * c.y);
  }
};

// 1 / d in FP64: the FP32 reciprocal (24 bits) and two Newton steps
// r <- r (2 - d r), each of which doubles the correct bits; the division
// outside 2^-99 <= |d| < 2^100, which FP32 holds with room.  The reciprocal heads
// every sweep's chain of dependent FP64 operations, of which a comparison is one
// too, so the range is told from the exponent.  An infinite pivot is no number to
// go on with: 1 / d = 0 would leave finite entries everywhere and hide it.
__device__ __forceinline__ double recip(double d) {
  const unsigned e = (unsigned)__double2hiint(d) >> 20 & 0x7ffu;
  if (e - 924u >= 199u) return e == 0x7ffu ? d - d : 1.0 / d;
  double r = (double)(1.0f / (float)d);
  r = fma(r, fma(-d, r, 1.0), r);
  return fma(r, fma(-d, r, 1.0), r);
}

// Inverse of the nb x nb block held two entries per thread (row tid / 8,
// columns 2 (tid % 8) and the next), by Gauss-Jordan sweeps.  Each sweep
// publishes row and column p and 1 / d as they are before it (the owner of
// the next diagonal entry takes the reciprocal as soon as it is updated).
// Returns false when a pivot is not positive (general: vanishes).
struct PivotSmem {
  double2 row[2][kNB], col[2][kNB], dinv[2];
  int bad[2];
};
template <bool general>
__device__ __forceinline__ bool pivot_inverse(double2 (&x)[2], int nb, PivotSmem& sm) {
  const int r = threadIdx.x >> 3, c0 = (threadIdx.x & 7) * 2;
  if (threadIdx.x < 2) sm.bad[threadIdx.x] = 0;
  __syncthreads();
  auto publish = [&](int p, int b) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int c = c0 + u;
      if (r == p && c == p) {
        const double2 d = x[u];
        if (general) {
          const double mag = d.x * d.x + d.y * d.y;
          if (!(mag > 1e-300)) sm.bad[b] = 1;
          const double inv = recip(mag);
          sm.dinv[b] = make_double2(d.x * inv, -d.y * inv);
        } else {   // Hermitian positive definite: real positive pivots
          if (!(d.x > 1e-150)) sm.bad[b] = 1;
          sm.dinv[b] = make_double2(recip(d.x), 0.0);
        }
      }
      if (r == p) sm.row[b][c] = x[u];
      if (c == p) sm.col[b][r] = x[u];
    }
  };
  publish(0, 0);
  for (int p = 0; p < nb; ++p) {
    const int b = p & 1;
    __syncthreads();
    if (sm.bad[b]) return false;   // one step's flag: the owner may already be setting the next
    const double2 di = sm.dinv[b], cr = sm.col[b][r];
    // every entry as x - f row_c: a_ij - (a_ip / d) a_pj; row p: 0 + a_pj / d;
    // column p: 0 - a_ip / d; the pivot: 0 + 1 / d (one path for all lanes:
    // a divergent FP64 instruction costs as much as a full one)
    double2 f = general ? cmul(cr, di) : make_double2(cr.x * di.x, cr.y * di.x);
    if (r == p) f = make_double2(-di.x, -di.y);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int c = c0 + u;
      const double2 rv = c == p ? make_double2(1.0, 0.0) : sm.row[b][c];
      if (r == p || c == p) x[u] = make_double2(0.0, 0.0);
      cmsub(x[u], f, rv);
    }
    if (p + 1 < nb) publish(p + 1, b ^ 1);
  }
  return true;
}

__device__ __forceinline__ void put_pivot(const double2 (&x)[2], double2* __restrict__ P) {
  const int r = threadIdx.x >> 3, c0 = (threadIdx.x & 7) * 2;
  P[r * kNB + c0] = x[0];
  P[r * kNB + c0 + 1] = x[1];
}

// P of the first block; a matrix of at most 16 rows is done with it.
template <bool full>
__global__ void __launch_bounds__(kThreads)
k_gj_first(Mats m, int nb, double2* __restrict__ pinv, int* __restrict__ err) {
  __shared__ PivotSmem sm;
  const int iw = blockIdx.x;
  const int r = threadIdx.x >> 3, c0 = (threadIdx.x & 7) * 2;
  double2 x[2];
#pragma unroll
  for (int u = 0; u < 2; ++u)
    x[u] = r < nb && c0 + u < nb ? m.get(iw, r, c0 + u, true) : make_double2(0.0, 0.0);
  if (!pivot_inverse<full>(x, nb, sm)) {
    if (threadIdx.x == 0) atomicExch(err, 1);
    return;
  }
  if (m.ng <= kNB) {
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (r < nb && c0 + u < nb) m.A[(size_t)iw * m.ng * m.ng + r * m.ng + c0 + u] = x[u];
  } else {
    put_pivot(x, pinv + (size_t)iw * 2 * kNB * kNB);
  }
}

// colpanel[iw][k][i] = A_i,b0+k (all i);  rowpanel[iw][k][j] = sum_l P_kl A_b0+l,j (all j).
// Entries above the diagonal tiles are not maintained; they follow from the
// stored ones: A_i,b = -conj(A_b,i) for i < b0 (i swept, b not), and
// A_b,j = conj(A_j,b) for j beyond the pivot block (neither swept).
// One thread per (column e, k), eight columns per block: the panels of one
// matrix spread over ng / 8 blocks (the FP64 rate of a single SM is low, and
// this step sits on the critical path of every pivot block).
template <bool full>
__global__ void __launch_bounds__(kThreads)
k_gj_panels(Mats m, int b0, int nb, const double2* __restrict__ pinv, double2* __restrict__ colp,
            double2* __restrict__ rowp) {
  __shared__ double2 base[kPE][kNB];  // A_b0+l,e of the block's columns
  const int iw = blockIdx.y, ng = m.ng;
  const bool first = b0 == 0;
  const double2* P = pinv + ((size_t)iw * 2 + ((b0 / kNB) & 1)) * kNB * kNB;
  double2* cp = colp + (size_t)iw * ng * kNB;
  double2* rp = rowp + (size_t)iw * kNB * ng;
  const int k = threadIdx.x & (kNB - 1), jj = threadIdx.x / kNB;
  const int e = blockIdx.x * kPE + jj;
  const bool live = e < ng && k < nb;
  if (live) {
    double2 v;
    if (full || e >= b0) {
      v = m.get(iw, e, b0 + k, first);
    } else {
      const double2 u = m.get(iw, b0 + k, e, first);
      v = make_double2(-u.x, u.y);
    }
    cp[(size_t)k * ng + e] = v;
    base[jj][k] = (full || e < b0 + nb) ? m.get(iw, b0 + k, e, first) : make_double2(v.x, -v.y);
  }
  __syncthreads();
  if (!live) return;
  double2 acc = make_double2(0.0, 0.0);
  for (int l = 0; l < nb; ++l) cmac(acc, P[k * kNB + l], base[jj][l]);
  rp[(size_t)k * ng + e] = acc;
}

// Update with block b0, and the pivot of the next block.  Blocks 0 .. nw - 1
// take the next diagonal tile of their matrix: updated, inverted, and written
// as P of the next step only (nothing else reads that tile in between).  The
// other blocks take the remaining 16 x 16 tiles in turn, each warp a quadrant
// (two entries of a row per lane), so that an SM's four FP64 units share every
// tile and the last one costs a quarter of what a tile per warp does.  The
// panels come straight from L1/L2: three loads of 16 bytes for eight
// multiply-adds, which take a warp's unit 512 clocks.  At most 40 registers:
// twelve blocks per SM hide the loads of a large matrix (96% of the FP64 rate at
// N_G = 3000, 88% with two), and two fit beside a tensor-core contraction block,
// so that the Dyson step of one frequency uses the FP64 units while the
// contraction of the next occupies the tensor cores.
template <bool full>
__global__ void __launch_bounds__(kThreads, 12)
k_gj_update(Mats m, int nw, int b0, int nb, double2* __restrict__ pinv, const double2* __restrict__ colp,
            const double2* __restrict__ rowp, int* __restrict__ err) {
  __shared__ PivotSmem sm;
  const int ng = m.ng;
  const int nt = (ng + kNB - 1) / kNB, pt = b0 / kNB;
  const bool first = b0 == 0, last = pt + 1 == nt;
  const size_t n2 = (size_t)ng * ng;
  int wb = blockIdx.x, workers = gridDim.x;
  if (!last) {
    if (wb < nw) {   // the next pivot
      const int iw = wb, r0 = (pt + 1) * kNB, nbn = min(kNB, ng - r0);
      const int r = threadIdx.x >> 3, c0 = (threadIdx.x & 7) * 2;
      const double2* ca = colp + (size_t)iw * kNB * ng + r0 + r;
      const double2* rb = rowp + (size_t)iw * kNB * ng + r0 + c0;
      double2 x[2];
#pragma unroll
      for (int u = 0; u < 2; ++u)
        x[u] = r < nbn && c0 + u < nbn ? m.get(iw, r0 + r, r0 + c0 + u, first) : make_double2(0.0, 0.0);
      if (r < nbn)
        for (int k = 0; k < nb; ++k) {
          const double2 a = ca[(size_t)k * ng];
#pragma unroll
          for (int u = 0; u < 2; ++u)
            if (c0 + u < nbn) cmsub(x[u], a, rb[(size_t)k * ng + u]);
        }
      if (!pivot_inverse<full>(x, nbn, sm)) {
        if (threadIdx.x == 0) atomicExch(err, 1);
        return;
      }
      put_pivot(x, pinv + ((size_t)iw * 2 + ((pt + 1) & 1)) * kNB * kNB);
      return;
    }
    wb -= nw;
    workers -= nw;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int lr = (warp >> 1) * 8 + (lane >> 2), lc = (warp & 1) * 8 + (lane & 3) * 2;   // row, first column
  const int per = full ? nt * nt : nt * (nt + 1) / 2;
  for (int t = wb; t < per * nw; t += workers) {
    const int iw = t / per, tile = t - iw * per;
    int I, J;
    if (full) {
      I = tile / nt;
      J = tile - I * nt;
    } else {
      I = (int)((sqrtf(8.0f * (float)tile + 1.0f) - 1.0f) * 0.5f);
      while ((I + 1) * (I + 2) / 2 <= tile) ++I;
      while (I * (I + 1) / 2 > tile) --I;
      J = tile - I * (I + 1) / 2;
    }
    if (!last && I == pt + 1 && J == pt + 1) continue;
    const int i = I * kNB + lr, j = J * kNB + lc;
    if (i >= ng || j >= ng) continue;
    const bool two = j + 1 < ng;   // a column beyond the matrix repeats the last
    // columns j, j + 1 of the row panel, or of P in the pivot columns
    const double2* rp = J == pt ? pinv + ((size_t)iw * 2 + (pt & 1)) * kNB * kNB + lc : rowp + (size_t)iw * kNB * ng + j;
    const int rld = J == pt ? kNB : ng;
    double2 x0 = make_double2(0.0, 0.0), x1 = x0;   // pivot columns: -A_ib P
    if (I == pt) {                                  // pivot rows: P A_bj; pivot block: P
      x0 = rp[lr * rld];
      if (two) x1 = rp[lr * rld + 1];
    } else {
      if (J != pt) {                                // elsewhere: A_ij - A_ib (P A_bj)
        x0 = m.get(iw, i, j, first);
        if (two) x1 = m.get(iw, i, j + 1, first);
      }
      const double2* cp = colp + (size_t)iw * kNB * ng + i;
      const int c1 = two ? 1 : 0;
#pragma unroll 2
      for (int k = 0; k < nb; ++k) {
        const double2 a = cp[k * ng];
        const double2 r0 = rp[k * rld], r1 = rp[k * rld + c1];
        cmsub(x0, a, r0);
        cmsub(x1, a, r1);
      }
    }
    double2* Am = m.A + iw * n2;
    Am[(size_t)i * ng + j] = x0;
    if (two) Am[(size_t)i * ng + j + 1] = x1;
    if (last && !full && I > J) {
      Am[(size_t)j * ng + i] = make_double2(x0.x, -x0.y);
      if (two) Am[(size_t)(j + 1) * ng + i] = make_double2(x1.x, -x1.y);
    }
  }
}

}  // namespace

// 54 clocks of an SM's FP64 units per 16 x 16 tile
double dyson_update_seconds(int ng, bool general) {
  const double nt = (ng + kNB - 1) / kNB;
  return 54.0 * (general ? nt * nt : 0.5 * nt * (nt + 1.0)) / 1.93e9;
}

namespace {

template <bool full>
cudaError_t launch_gj(const Mats& m, int nw, double2* colp, double2* rowp, double2* pinv, int* err, cudaStream_t s,
                      bool beside) {
  const int ng = m.ng, nt = (ng + kNB - 1) / kNB;
  // Blocks of the update, fewer when there are fewer tiles.  As many per SM as its
  // registers allow hide the loads best, but the next pivot shares its SM's FP64
  // units with them and has to end before they do.  Alone that is so from five times
  // the chain on (four matrices of N_G = 3000 420 -> 382 ms against two per SM, three
  // of 1000 12.2 -> 11.7; two of 900 6.32 ms with two, 6.57 with twelve, three of 431
  // 1.40 and 1.54).  Beside a contraction, where two groups share the SMs, from one
  // matrix as long as the chain on (two of N_G = 750 4.15 -> 3.80 ms, the precision
  // workload on 6x6x6 k 291 -> 282, six of N_G = 3000 664 -> 583); below, a contraction
  // cannot start while blocks of the higher-priority Dyson step wait (nine metals of
  // N_G = 178 to 330 in a batch 15.4 ms with two, 16.6 with twelve).
  const double work = dyson_update_seconds(ng, full);
  const bool longer = beside ? work >= kDysonChain : work * nw >= 5.0 * kDysonChain;
  const int most = (longer ? 12 : 2) * 152;
  k_gj_first<full><<<nw, kThreads, 0, s>>>(m, ng < kNB ? ng : kNB, pinv, err);
  if (nt > 1)
    for (int b0 = 0; b0 < ng; b0 += kNB) {
      const int nb = ng - b0 < kNB ? ng - b0 : kNB;
      const bool last = b0 + kNB >= ng;
      k_gj_panels<full><<<dim3((ng + kPE - 1) / kPE, nw), kThreads, 0, s>>>(m, b0, nb, pinv, colp, rowp);
      const int64_t tiles = (int64_t)(full ? nt * nt : nt * (nt + 1) / 2) * nw;
      const int spare = last ? most : nw < most / 2 ? most - nw : most / 2;
      const int workers = (int)(tiles < spare ? tiles : spare);
      k_gj_update<full><<<workers + (last ? 0 : nw), kThreads, 0, s>>>(m, nw, b0, nb, pinv, colp, rowp, err);
    }
  return cudaGetLastError();
}

}  // namespace

int dyson_launches(int ng) {
  const int nt = (ng + kNB - 1) / kNB;
  return nt > 1 ? 1 + 2 * nt : 1;
}

cudaError_t dyson_prepare() {
  const void* fns[] = {(const void*)k_gj_first<false>,  (const void*)k_gj_first<true>,
                       (const void*)k_gj_panels<false>, (const void*)k_gj_panels<true>,
                       (const void*)k_gj_update<false>, (const void*)k_gj_update<true>};
  for (const void* f : fns) {
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout,
                                               cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_dyson(const double2* chi, const double* vsqrt, int ng, int nw, double2* A,
                         double2* colp, double2* rowp, double2* pinv, int* err, cudaStream_t s, bool beside) {
  return launch_gj<false>(Mats{chi, vsqrt, A, ng}, nw, colp, rowp, pinv, err, s, beside);
}

// General (non-Hermitian) eps~ of real-axis frequencies: the same blocked
// Gauss-Jordan over every tile, reading A directly, with no mirror.
// Pivoting is not needed there: for w > 0 with eta > 0 every weight's
// imaginary part is <= 0, so eps~ has a positive semidefinite imaginary
// (anti-Hermitian) part, which every Schur complement inherits; a pivot that
// vanishes all the same is reported through the error flag.
cudaError_t launch_dyson_general(const double2* chi, const double* vsqrt, int ng, int nw, double2* A,
                                 double2* colp, double2* rowp, double2* pinv, int* err, cudaStream_t s, bool beside) {
  return launch_gj<true>(Mats{chi, vsqrt, A, ng}, nw, colp, rowp, pinv, err, s, beside);
}

}  // namespace chi0
