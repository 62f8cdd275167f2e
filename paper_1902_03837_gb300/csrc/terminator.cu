// Learned band-sum terminator: a small network predicts the contribution of
// the bands left out of a truncated chi0.
//
// The paper corrects a band-truncated chi0 with the Bruneval-Gonze
// X-terminator (Eq. X_term_def, Appendix C): chi0 = chi0^trunc + Delta chi.
// Here Delta chi_{GG'}(w) is predicted per matrix entry from the features
//     x = (|q+G| / Kn, |q+G'| / Kn, Im w / Wn, Re chi0^trunc / c, Im chi0^trunc / c)
// (Kn = largest |q+G| of the response set, Wn = largest |Im w|, c = mean
// |chi0^trunc_GG(w_0)|), and the prediction c (y_0 + i y_1) is Hermitised
// before it is added.  The network: h1 = tanh(W1 x + b1), h2 = tanh(W2 h1 +
// b2), y = W3 h2 + b3 (5 -> 128 -> 128 -> 2); parameters packed as W1, b1,
// W2, b2, W3, b3 in FP32 (master copy).  In BF16 mode every matrix product
// takes BF16-rounded operands and accumulates in FP32.  Training: loss
// L = 1/(2B) sum (y - t)^2, gradients by backpropagation, Adam updates.
#include <cuda_bf16.h>

#include <cmath>
#include <vector>

#include "ctx.cuh"

namespace chi0 {

namespace {

constexpr int kI = 5, kH = 128, kO = 2;
constexpr int kP = kH * kI + kH + kH * kH + kH + kO * kH + kO;  // 17538
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kH * kI, kOffW2 = kOffB1 + kH, kOffB2 = kOffW2 + kH * kH,
              kOffW3 = kOffB2 + kH, kOffB3 = kOffW3 + kO * kH;
constexpr int kS = 32;         // samples per block of the training kernel
constexpr int kSP = 64;        // samples per pass of the prediction kernel
constexpr int kThreads = 256;
constexpr int kTrainThreads = 512;
constexpr int kLd = kH + 4;    // padded row: eight rows' 16-byte pieces fall into distinct banks

__device__ __forceinline__ float rb(float v, int bf16) {
  return bf16 ? __bfloat162float(__float2bfloat16_rn(v)) : v;
}

// acc[i][j] += sum_k A[s_i][k] B[h_j][k], k ascending (rows of kLd floats in
// shared memory; s_i = 8 i + lane / 4, h_j = 32 j + 4 (warp % 8) + lane % 4).  Both
// layers of the network are bound by the FP32 pipe once the operands come as
// 16-byte pieces for NS x 4 outputs per thread (one load per 2 NS x 8 / (NS + 4)
// multiply-adds; a scalar pair of loads per multiply-add was bound by shared
// memory).  Every output keeps its own chain of fused multiply-adds in the
// order of k, so the results do not depend on the tiling.
template <int NS>
__device__ __forceinline__ void rows_dot(const float* __restrict__ A, const float* __restrict__ B, float (&acc)[NS][4]) {
  const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) & 7;
  const float* a = A + (lane >> 2) * kLd;
  const float* b = B + (warp * 4 + (lane & 3)) * kLd;
#pragma unroll 2
  for (int k = 0; k < kH; k += 4) {
    float4 av[NS], bv[4];
#pragma unroll
    for (int i = 0; i < NS; ++i) av[i] = *reinterpret_cast<const float4*>(a + i * 8 * kLd + k);
#pragma unroll
    for (int j = 0; j < 4; ++j) bv[j] = *reinterpret_cast<const float4*>(b + j * 32 * kLd + k);
#pragma unroll
    for (int i = 0; i < NS; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        acc[i][j] = fmaf(bv[j].x, av[i].x, acc[i][j]);
        acc[i][j] = fmaf(bv[j].y, av[i].y, acc[i][j]);
        acc[i][j] = fmaf(bv[j].z, av[i].z, acc[i][j]);
        acc[i][j] = fmaf(bv[j].w, av[i].w, acc[i][j]);
      }
  }
}

// The parameters as every pass of a block uses them: products' operands rounded.
struct alignas(16) MlpWeights {
  alignas(16) float W2[kH * kLd];
  alignas(16) float w3[kO * kH];
  float w1[kH * kI], b1[kH], b2[kH], b3[kO];
};
template <int NT>   // threads of the block
__device__ __forceinline__ void load_weights(MlpWeights& w, const float* __restrict__ prm, int bf16) {
  const int tid = threadIdx.x;
#pragma unroll 16
  for (int e = tid; e < kH * kH; e += NT)   // (the caller's vector is only 4-byte aligned)
    w.W2[(e / kH) * kLd + e % kH] = rb(prm[kOffW2 + e], bf16);
  for (int e = tid; e < kH * kI; e += NT) w.w1[e] = rb(prm[kOffW1 + e], bf16);
  for (int e = tid; e < kO * kH; e += NT) w.w3[e] = rb(prm[kOffW3 + e], bf16);
  if (tid < kH) {
    w.b1[tid] = prm[kOffB1 + tid];
    w.b2[tid] = prm[kOffB2 + tid];
  }
  if (tid < kO) w.b3[tid] = prm[kOffB3 + tid];
}

__device__ __forceinline__ float layer1(const MlpWeights& w, const float* __restrict__ xs, int s, int h) {
  float z = w.b1[h];
#pragma unroll
  for (int i = 0; i < kI; ++i) z = fmaf(w.w1[h * kI + i], xs[s * kI + i], z);
  return tanhf(z);
}

// y[s][o] of rows h2[s] (rounded)
__device__ __forceinline__ float layer3(const MlpWeights& w, const float* __restrict__ h2, int s, int o) {
  float z = w.b3[o];
#pragma unroll 4
  for (int k = 0; k < kH; k += 4) {
    const float4 a = *reinterpret_cast<const float4*>(h2 + s * kLd + k);
    const float4 b = *reinterpret_cast<const float4*>(w.w3 + o * kH + k);
    z = fmaf(b.x, a.x, z);
    z = fmaf(b.y, a.y, z);
    z = fmaf(b.z, a.z, z);
    z = fmaf(b.w, a.w, z);
  }
  return z;
}

// Prediction with FP32 operands: two blocks per SM stay for the whole launch and
// take kSP samples at a time, so that the parameters are staged once per block.
// Bound by the FP32 pipe (17.3 k multiply-adds and 256 tanh per sample): 10^6
// samples 5180 -> 929 us (0.67 ms of issue slots).
struct PredictSmem {
  MlpWeights w;
  alignas(16) float h[kSP * kLd];
  float xs[kSP * kI];
};
__global__ void __launch_bounds__(kThreads, 2)
k_mlp_predict(const float* __restrict__ prm, const float* __restrict__ x, int64_t batch, float* __restrict__ y) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PredictSmem& sm = *reinterpret_cast<PredictSmem*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  load_weights<kThreads>(sm.w, prm, 0);
  for (int64_t s0 = (int64_t)blockIdx.x * kSP; s0 < batch; s0 += (int64_t)gridDim.x * kSP) {
    const int ns = (int)min((int64_t)kSP, batch - s0);
    for (int e = tid; e < kSP * kI; e += kThreads) sm.xs[e] = e < ns * kI ? x[s0 * kI + e] : 0.f;
    __syncthreads();
    for (int s = tid / kH; s < kSP; s += kThreads / kH) sm.h[s * kLd + tid % kH] = layer1(sm.w, sm.xs, s, tid % kH);
    __syncthreads();
    float acc[kSP / 8][4];
#pragma unroll
    for (int i = 0; i < kSP / 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = sm.w.b2[j * 32 + warp * 4 + (lane & 3)];
    rows_dot(sm.h, sm.w.W2, acc);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kSP / 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j)
        sm.h[(i * 8 + (lane >> 2)) * kLd + j * 32 + warp * 4 + (lane & 3)] = tanhf(acc[i][j]);
    __syncthreads();
    if (tid < kSP * kO) {
      const int s = tid % kSP, o = tid / kSP;
      const float z = layer3(sm.w, sm.h, s, o);
      if (s < ns) y[(s0 + s) * kO + o] = z;
    }
    // the next pass writes xs (read before the last barrier but one) and h
    // (behind its own first barrier)
  }
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ float low_bf16(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float high_bf16(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }
// c += a b^T, 16 x 8 x 16, BF16 operands, FP32 sums.  With g = lane / 4 and t =
// lane % 4: a = rows g, g + 8 at k = 2t, 2t + 1, then both at k + 8; b = row g at
// the same k; c = rows g, g + 8 at columns 2t, 2t + 1.
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// four 8 x 8 matrices of BF16 (lane l gives the address of row l % 8 of matrix
// l / 8): lane l gets row l / 4, columns 2 (l % 4), + 1 of each
__device__ __forceinline__ void ldsm(uint32_t (&r)[4], const __nv_bfloat16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p))
               : "memory");
}

// Prediction with BF16 operands: the 128 x 128 layer on the tensor cores.  A warp
// takes 16 samples from input to output without a barrier: its lanes compute the
// first layer where the matrix instruction wants the operand and the last one
// where it leaves the sums.  256 tanh and 900 multiply-adds per sample remain on
// the FP32 pipe and bound the kernel, not the matrix product (so the register
// form of the instruction does, and TMEM's extra trips would not be hidden).
//
// h2 = bf16(tanh(z)) keeps the value that the chain of FP32 multiply-adds in the
// order of k gives (as the training kernel computes it): the tensor core's z
// differs from the chain's by its rounding only, so the two can round apart
// only next to a rounding boundary.  Where z +- kDoubt P straddles one, the value
// goes on a list, and the chain is run for up to 32 of the list at a time, one per
// lane.  Both roundings go with the size of the partial sums, the bias among them,
// and P bounds those: the largest |z| after any of the four steps of 32 terms, and
// half the largest sum of 32 |W2|, by which a sum can exceed both ends of its
// step.  128 roundings of half an ulp add up to 3.3 ulp in the mean where all
// partial sums are equally large (a bias of 0.6 and small weights), and the tensor
// core drops up to one per 16 terms.  Over 8.4 million values each of eleven
// networks (initial, trained-like, biases far above the weights, sums that rise
// and fall) the two differ by 15 2^-23 of the largest partial sum at most, by
// 0.2-3 in the root mean square, so kDoubt is 16 2^-23: none of their values went
// unnoticed.  (With 2^-23 sum |W2| for kDoubt P up to 133 did, where a bias was
// above the weights.)  Some 25 of a warp's 2048 values are listed.
// 10^6 samples: 929 us on the FP32 pipe -> 424 us (0.26 ms of issue slots; 352 with
// the narrower doubt, which lists 14).
constexpr float kDoubt = 1.f / 524288.f;
constexpr int kTrack = 2;           // products of 16 terms between looks at the sums
constexpr int kLdb = kH + 8;        // padded row of BF16: eight rows' 16-byte pieces fall into distinct banks
constexpr int kPredWarps = 8;
constexpr int kList = 32 + 128;     // below 32 before a step, which adds 128 at most
struct PredictBf16Smem {
  alignas(16) __nv_bfloat16 w2[kH * kLdb];
  alignas(16) __nv_bfloat16 h1[kPredWarps][16 * kLdb];
  float4 w1[kH];                    // inputs 0..3
  float4 w3[kH / 2];                // both outputs' weights of two inputs
  float2 w1b[kH];                   // input 4, bias
  float2 b2[kH / 2], doubt[kH / 2];   // doubt: kDoubt / 2 of the largest sum of 32 |W2|
  uint32_t list[kPredWarps][kList]; // h2 as the tensor core's z gives it | sample | column
};
static_assert(kPredWarps * 32 == kThreads, "a warp per tile");
__global__ void __launch_bounds__(kThreads, 2)
k_mlp_predict_bf16(const float* __restrict__ prm, const float* __restrict__ x, int64_t batch, float* __restrict__ y) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PredictBf16Smem& sm = *reinterpret_cast<PredictBf16Smem*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
#pragma unroll 8
  for (int e = tid; e < kH * kH; e += kThreads) sm.w2[(e / kH) * kLdb + e % kH] = __float2bfloat16_rn(prm[kOffW2 + e]);
  if (tid < kH) {
    const float* w = prm + kOffW1 + tid * kI;
    sm.w1[tid] = make_float4(rb(w[0], 1), rb(w[1], 1), rb(w[2], 1), rb(w[3], 1));
    sm.w1b[tid] = make_float2(rb(w[4], 1), prm[kOffB1 + tid]);
  } else if (tid < kH + kH / 2) {
    const int p = tid - kH;
    const float* w = prm + kOffW3 + 2 * p;
    sm.w3[p] = make_float4(rb(w[0], 1), rb(w[1], 1), rb(w[kH], 1), rb(w[kH + 1], 1));
    sm.b2[p] = make_float2(prm[kOffB2 + 2 * p], prm[kOffB2 + 2 * p + 1]);
  }
  const float b3 = prm[kOffB3 + (t & 1)];
  __syncthreads();
  if (tid < kH) {
    float most = 0.f;
    for (int k = 0; k < kH; k += 16 * kTrack) {
      float s = 0.f;
      for (int q = 0; q < 16 * kTrack; ++q) s += fabsf(__bfloat162float(sm.w2[tid * kLdb + k + q]));
      most = fmaxf(most, s);
    }
    reinterpret_cast<float*>(sm.doubt)[tid] = 0.5f * kDoubt * most;
  }
  __syncthreads();
  __nv_bfloat16* h1s = sm.h1[warp];
  uint32_t* list = sm.list[warp];
  for (int64_t s0 = ((int64_t)blockIdx.x * kPredWarps + warp) * 16; s0 < batch;
       s0 += (int64_t)gridDim.x * kPredWarps * 16) {
    float xr[2][kI];   // rows g, g + 8 of the tile
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int i = 0; i < kI; ++i) xr[r][i] = s0 + g + 8 * r < batch ? rb(x[(s0 + g + 8 * r) * kI + i], 1) : 0.f;
    uint32_t a[kH / 16][4];
#pragma unroll
    for (int ks = 0; ks < kH / 16; ++ks)
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        float h[2][2];
        const int c0 = ks * 16 + half * 8 + t * 2;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const float4 w = sm.w1[c0 + j];
          const float2 wb = sm.w1b[c0 + j];
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            float z = fmaf(w.x, xr[r][0], wb.y);
            z = fmaf(w.y, xr[r][1], z);
            z = fmaf(w.z, xr[r][2], z);
            z = fmaf(w.w, xr[r][3], z);
            h[r][j] = tanhf(fmaf(wb.x, xr[r][4], z));
          }
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          a[ks][2 * half + r] = pack_bf16(h[r][0], h[r][1]);
          *reinterpret_cast<uint32_t*>(h1s + (g + 8 * r) * kLdb + c0) = a[ks][2 * half + r];
        }
      }
    float out[2][kO] = {};
    int n = 0;   // entries on the list
    // the chains of the last cnt entries; their h2 in place of the tensor core's
    auto settle = [&](int cnt) {
      __syncwarp();
      n -= cnt;
      float d = 0.f;
      int row = 0, col = 0;
      if (lane < cnt) {
        const uint32_t e = list[n + lane];
        row = (e >> 7) & 15;
        col = e & (kH - 1);
        float z = reinterpret_cast<const float*>(sm.b2)[col];
        const uint4* hp = reinterpret_cast<const uint4*>(h1s + row * kLdb);
        const uint4* wp = reinterpret_cast<const uint4*>(sm.w2 + col * kLdb);
#pragma unroll 4
        for (int k = 0; k < kH / 8; ++k) {
          const uint4 h = hp[k], w = wp[k];
          const uint32_t hv[4] = {h.x, h.y, h.z, h.w}, wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            z = fmaf(low_bf16(wv[q]), low_bf16(hv[q]), z);
            z = fmaf(high_bf16(wv[q]), high_bf16(hv[q]), z);
          }
        }
        d = rb(tanhf(z), 1) - high_bf16(e);
      }
      for (uint32_t m = __ballot_sync(0xffffffffu, !(d == 0.f)); m; m &= m - 1) {
        const int b = __ffs(m) - 1;
        const int rr = __shfl_sync(0xffffffffu, row, b), cc = __shfl_sync(0xffffffffu, col, b);
        const float dd = __shfl_sync(0xffffffffu, d, b);
        const float* w = reinterpret_cast<const float*>(sm.w3 + (cc >> 1)) + (cc & 1);
        if (lane == (rr & 7) * 4) {
#pragma unroll
          for (int r = 0; r < 2; ++r)
            if (rr >> 3 == r) {
              out[r][0] = fmaf(w[0], dd, out[r][0]);
              out[r][1] = fmaf(w[2], dd, out[r][1]);
            }
        }
      }
      __syncwarp();
    };
    for (int n0 = 0; n0 < kH; n0 += 16) {
      float c[2][4], most[2][4];   // sums, and the largest of them so far
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float2 b2 = sm.b2[n0 / 2 + 4 * j + t];
        c[j][0] = c[j][2] = b2.x;
        c[j][1] = c[j][3] = b2.y;
#pragma unroll
        for (int q = 0; q < 4; ++q) most[j][q] = fabsf(c[j][q]);
      }
#pragma unroll
      for (int ks = 0; ks < kH / 16; ++ks) {
        uint32_t b[4];
        ldsm(b, sm.w2 + (n0 + (lane & 7) + (lane >> 4) * 8) * kLdb + ks * 16 + ((lane >> 3) & 1) * 8);
        mma_bf16(c[0], a[ks], b[0], b[1]);
        mma_bf16(c[1], a[ks], b[2], b[3]);
        if (ks % kTrack == kTrack - 1) {
#pragma unroll
          for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) most[j][q] = fmaxf(most[j][q], fabsf(c[j][q]));
        }
      }
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int p = n0 / 2 + 4 * j + t;
        const float4 w = sm.w3[p];
        const float2 dz = sm.doubt[p];
        uint32_t h[2], open[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const float h0 = tanhf(c[j][2 * r]), h1 = tanhf(c[j][2 * r + 1]);
          // the doubt times the slope of tanh, and an ulp for tanhf itself
          const float d0 = fmaf(kDoubt, most[j][2 * r], dz.x), d1 = fmaf(kDoubt, most[j][2 * r + 1], dz.y);
          const float e0 = fmaf(d0, fmaf(-h0, h0, 1.f), 1.2e-7f), e1 = fmaf(d1, fmaf(-h1, h1, 1.f), 1.2e-7f);
          h[r] = pack_bf16(h0, h1);
          open[r] = pack_bf16(h0 + e0, h1 + e1) ^ pack_bf16(h0 - e0, h1 - e1);
          const float r0 = low_bf16(h[r]), r1 = high_bf16(h[r]);
          out[r][0] = fmaf(w.y, r1, fmaf(w.x, r0, out[r][0]));
          out[r][1] = fmaf(w.w, r1, fmaf(w.z, r0, out[r][1]));
        }
        if (__any_sync(0xffffffffu, (open[0] | open[1]) != 0)) {
#pragma unroll
          for (int v = 0; v < 4; ++v) {   // row g + 8 (v / 2), column 2 p + v % 2
            const uint32_t o = v & 1 ? open[v >> 1] >> 16 : open[v >> 1] & 0xffffu;
            const uint32_t m = __ballot_sync(0xffffffffu, o != 0);
            if (o != 0)
              list[n + __popc(m & ((1u << lane) - 1))] =
                  (v & 1 ? h[v >> 1] & 0xffff0000u : h[v >> 1] << 16) | (uint32_t)((g + 8 * (v >> 1)) << 7) |
                  (uint32_t)(2 * p + (v & 1));
            n += __popc(m);
          }
          while (n >= 32) settle(32);
        }
      }
    }
    if (n > 0) settle(n);
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int o = 0; o < kO; ++o) {
        out[r][o] += __shfl_xor_sync(0xffffffffu, out[r][o], 1);
        out[r][o] += __shfl_xor_sync(0xffffffffu, out[r][o], 2);
      }
    // lane t writes output t % 2 of row g + 8 (t / 2)
    const float lo = t & 1 ? out[0][1] : out[0][0], hi = t & 1 ? out[1][1] : out[1][0];
    const int64_t row = s0 + g + 8 * (t >> 1);
    if (row < batch) y[row * kO + (t & 1)] = (t & 2 ? hi : lo) + b3;
    __syncwarp();   // h1 of the next tile
  }
}

// Forward and backward for kS samples per block.  Gradients of the block go to
// part[block][kP] (summed later in a fixed order).  Per-sample values are the
// same chains as in the prediction; the three products of 32 x 128 x 128 (h2,
// dz1, dW2) take 2 x 4, 2 x 4 and 8 x 4 outputs per thread.  A block holds an SM
// (one per SM at the minibatch of 4096), so its own 16 warps have to cover the
// latencies: a training step there, with the reduction and Adam, 91.7 us -> 36.8
// with 8 warps and twice the outputs per thread -> 34.8 us.
struct TrainSmem {
  MlpWeights w;
  alignas(16) float h1[kS * kLd], h2[kS * kLd], d2[kS * kLd], d1[kS * kLd];   // rounded operands
  alignas(16) float r2[kS * kLd], r1[kS * kLd];                               // dz2, dz1 as computed
  float xs[kS * kI], ys[kS * kO], red[32];
};
__global__ void __launch_bounds__(kTrainThreads, 1)
k_mlp_train(const float* __restrict__ prm, const float* __restrict__ x, const float* __restrict__ t, int64_t batch,
            int bf16, float* __restrict__ part, float* __restrict__ loss_part) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TrainSmem& sm = *reinterpret_cast<TrainSmem*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t s0 = (int64_t)blockIdx.x * kS;
  const int ns = (int)min((int64_t)kS, batch - s0);
  load_weights<kTrainThreads>(sm.w, prm, bf16);
  for (int e = tid; e < kS * kI; e += kTrainThreads) sm.xs[e] = e < ns * kI ? rb(x[s0 * kI + e], bf16) : 0.f;
  __syncthreads();
  const int r0 = (warp >> 3) * 16, sr = r0 + (lane >> 2);   // rows sr + 8 i of the warp's half
  const int hc = (warp & 7) * 4 + (lane & 3);               // layer 2: columns hc + 32 j
  const int kc = hc * 4;                                    // layer 1: columns kc + j
  float h1v[2][4], h2v[2][4];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    float4 r;
#pragma unroll
    for (int j = 0; j < 4; ++j) h1v[i][j] = layer1(sm.w, sm.xs, sr + 8 * i, kc + j);
    r = make_float4(rb(h1v[i][0], bf16), rb(h1v[i][1], bf16), rb(h1v[i][2], bf16), rb(h1v[i][3], bf16));
    *reinterpret_cast<float4*>(sm.h1 + (sr + 8 * i) * kLd + kc) = r;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) h2v[i][j] = sm.w.b2[hc + 32 * j];
  rows_dot(sm.h1 + r0 * kLd, sm.w.W2, h2v);
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      h2v[i][j] = tanhf(h2v[i][j]);
      sm.h2[(sr + 8 * i) * kLd + hc + 32 * j] = rb(h2v[i][j], bf16);
    }
  __syncthreads();
  // layer 3, loss and dy = (y - t) / B
  float lsum = 0.f;
  if (tid < kS * kO) {
    const int s = tid / kO, o = tid % kO;
    float r = 0.f;
    if (s < ns) r = layer3(sm.w, sm.h2, s, o) - t[(s0 + s) * kO + o];
    lsum = r * r;
    sm.ys[tid] = r / (float)batch;
  }
  if (warp == 1) sm.red[lane] = lsum;
  __syncthreads();
  if (warp == 0) {   // kS kO = 64 values
    lsum += sm.red[lane];
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, w);
    if (lane == 0) loss_part[blockIdx.x] = 0.5f * lsum / (float)batch;
  }
  // dz2 = (dy W3) * (1 - h2^2)
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int s = sr + 8 * i, h = hc + 32 * j;
      float g = 0.f;
#pragma unroll
      for (int o = 0; o < kO; ++o) g = fmaf(rb(sm.ys[s * kO + o], bf16), sm.w.w3[o * kH + h], g);
      const float hv = h2v[i][j];
      const float d = s < ns ? g * (1.f - hv * hv) : 0.f;
      sm.r2[s * kLd + h] = d;
      sm.d2[s * kLd + h] = rb(d, bf16);
    }
  __syncthreads();
  // dz1 = (dz2 W2) * (1 - h1^2), h ascending
  {
    float g[2][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) g[i][j] = 0.f;
#pragma unroll 2
    for (int h = 0; h < kH; h += 4) {
      float4 dv[2], wv[4];
#pragma unroll
      for (int i = 0; i < 2; ++i) dv[i] = *reinterpret_cast<const float4*>(sm.d2 + (sr + 8 * i) * kLd + h);
#pragma unroll
      for (int q = 0; q < 4; ++q) wv[q] = *reinterpret_cast<const float4*>(sm.w.W2 + (h + q) * kLd + kc);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float dq[4] = {dv[i].x, dv[i].y, dv[i].z, dv[i].w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          g[i][0] = fmaf(dq[q], wv[q].x, g[i][0]);
          g[i][1] = fmaf(dq[q], wv[q].y, g[i][1]);
          g[i][2] = fmaf(dq[q], wv[q].z, g[i][2]);
          g[i][3] = fmaf(dq[q], wv[q].w, g[i][3]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int s = sr + 8 * i;
      float d[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float hv = h1v[i][j];
        d[j] = s < ns ? g[i][j] * (1.f - hv * hv) : 0.f;
      }
      *reinterpret_cast<float4*>(sm.r1 + s * kLd + kc) = make_float4(d[0], d[1], d[2], d[3]);
      *reinterpret_cast<float4*>(sm.d1 + s * kLd + kc) =
          make_float4(rb(d[0], bf16), rb(d[1], bf16), rb(d[2], bf16), rb(d[3], bf16));
    }
  }
  __syncthreads();
  float* gp = part + (size_t)blockIdx.x * kP;
  // dW2[h][k] = sum_s dz2[s][h] h1[s][k]
  {
    const int h0 = (tid >> 5) * 8, k0 = lane * 4;
    float g[8][4];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) g[a][b] = 0.f;
#pragma unroll 4
    for (int s = 0; s < kS; ++s) {
      const float4 d0 = *reinterpret_cast<const float4*>(sm.d2 + s * kLd + h0);
      const float4 d1 = *reinterpret_cast<const float4*>(sm.d2 + s * kLd + h0 + 4);
      const float4 a0 = *reinterpret_cast<const float4*>(sm.h1 + s * kLd + k0);
      const float d[8] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
      const float h[4] = {a0.x, a0.y, a0.z, a0.w};
#pragma unroll
      for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) g[a][b] = fmaf(d[a], h[b], g[a][b]);
    }
    if (((uintptr_t)gp & 7) == 0) {   // kP and kOffW2 are even: 8-byte pieces where the caller's buffer allows
#pragma unroll
      for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 4; b += 2)
          *reinterpret_cast<float2*>(gp + kOffW2 + (h0 + a) * kH + k0 + b) = make_float2(g[a][b], g[a][b + 1]);
    } else {
#pragma unroll
      for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) gp[kOffW2 + (h0 + a) * kH + k0 + b] = g[a][b];
    }
  }
  if (tid < 2 * kH) {
    // dW3[o][h] = sum_s dy[s][o] h2[s][h]
    const int o = tid / kH, h = tid % kH;
    float g = 0.f;
#pragma unroll 8
    for (int s = 0; s < kS; ++s) g = fmaf(rb(sm.ys[s * kO + o], bf16), sm.h2[s * kLd + h], g);
    gp[kOffW3 + tid] = g;
    // db2, db1
    const float* r = tid < kH ? sm.r2 : sm.r1;
    g = 0.f;
#pragma unroll 8
    for (int s = 0; s < kS; ++s) g += r[s * kLd + h];
    gp[(tid < kH ? kOffB2 : kOffB1) + h] = g;
  } else {
    // dW1[h][i] = sum_s dz1[s][h] x[s][i];  db3
    for (int e = tid - 2 * kH; e < kH * kI; e += kTrainThreads - 2 * kH) {
      const int h = e / kI, i = e % kI;
      float g = 0.f;
#pragma unroll 8
      for (int s = 0; s < kS; ++s) g = fmaf(sm.d1[s * kLd + h], sm.xs[s * kI + i], g);
      gp[kOffW1 + e] = g;
    }
    if (tid - 2 * kH < kO) {
      float g = 0.f;
      for (int s = 0; s < kS; ++s) g += sm.ys[s * kO + tid - 2 * kH];
      gp[kOffB3 + tid - 2 * kH] = g;
    }
  }
}
static_assert(sizeof(MlpWeights) % 16 == 0 && kLd % 4 == 0, "16-byte pieces");
static_assert(kS == 32 && kTrainThreads == 4 * kH && kO == 2, "thread maps of k_mlp_train");

// Sum of the block partials, block by block: the order is that of the samples,
// whatever their number.  32 loads of a thread are in flight; the chain of
// additions (128 at the minibatch of 4096, 0.3 us) is not what the kernel waits for.
constexpr int kRedP = 64;
__global__ void __launch_bounds__(kRedP)
k_mlp_reduce(const float* __restrict__ part, int nblk, const float* __restrict__ lpart, float* __restrict__ grad,
             float* __restrict__ loss) {
  const int p = blockIdx.x * kRedP + threadIdx.x;
  if (p > kP || (p == kP && !loss)) return;
  const float* src = p < kP ? part + p : lpart;
  const size_t stride = p < kP ? kP : 1;
  float g = 0.f;
  int b = 0;
  for (; b + 32 <= nblk; b += 32) {
    float v[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = src[(size_t)(b + i) * stride];
#pragma unroll
    for (int i = 0; i < 32; ++i) g += v[i];
  }
  for (; b < nblk; ++b) g += src[(size_t)b * stride];
  *(p < kP ? grad + p : loss) = g;
}

__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, int64_t n, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const float gk = g[k];
  const float mk = b1 * m[k] + (1.f - b1) * gk;
  const float vk = b2 * v[k] + (1.f - b2) * gk * gk;
  m[k] = mk;
  v[k] = vk;
  p[k] -= lr * (mk / c1) / (sqrtf(vk / c2) + eps);
}

}  // namespace

int mlp_nparams() { return kP; }

cudaError_t mlp_loss_grad(const float* prm, const float* x, const float* t, int64_t batch, int bf16,
                          float* grad, float* loss, float* part, float* lpart, cudaStream_t st) {
  const int nblk = (int)((batch + kS - 1) / kS);
  cudaError_t e = cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(TrainSmem));
  if (e != cudaSuccess) return e;
  k_mlp_train<<<nblk, kTrainThreads, sizeof(TrainSmem), st>>>(prm, x, t, batch, bf16, part, lpart);
  k_mlp_reduce<<<kP / kRedP + 1, kRedP, 0, st>>>(part, nblk, lpart, grad, loss);
  return cudaGetLastError();
}

cudaError_t mlp_predict(const float* prm, const float* x, int64_t batch, int bf16, float* y,
                        cudaStream_t st) {
  const int64_t rows = bf16 ? 16 * kPredWarps : kSP, passes = (batch + rows - 1) / rows;
  const size_t smem = bf16 ? sizeof(PredictBf16Smem) : sizeof(PredictSmem);
  auto kernel = bf16 ? k_mlp_predict_bf16 : k_mlp_predict;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kernel<<<(unsigned)(passes < 2 * 152 ? passes : 2 * 152), kThreads, smem, st>>>(prm, x, batch, y);
  return cudaGetLastError();
}

cudaError_t mlp_adam(float* p, const float* g, float* m, float* v, int64_t n, float lr, float b1,
                     float b2, float eps, int step, cudaStream_t st) {
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  k_adam<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(p, g, m, v, n, lr, b1, b2, eps, c1, c2);
  return cudaGetLastError();
}

}  // namespace chi0

// ---------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------
namespace chi0 {
namespace {

// c = mean |chi_ii(w_0)| and 1/c (device, no host round trip)
__global__ void k_diag_scale(const double2* __restrict__ chi, int ng, double* __restrict__ out) {
  __shared__ double red[256];
  double s = 0.0;
  for (int i = threadIdx.x; i < ng; i += 256) {
    const double2 v = chi[(size_t)i * ng + i];
    s += sqrt(v.x * v.x + v.y * v.y);
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double c = red[0] / ng;
    out[0] = c > 0.0 ? c : 1.0;
    out[1] = 1.0 / out[0];
  }
}

__global__ void k_term_features_dev(const double2* __restrict__ chi, const double2* __restrict__ full,
                                    const double* __restrict__ qgn, const double* __restrict__ wn,
                                    int ng, int nw, const double* __restrict__ cs, float* __restrict__ x,
                                    float* __restrict__ t) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t n2 = (int64_t)ng * ng;
  if (e >= n2 * nw) return;
  const double inv_c = cs[1];
  const int iw = (int)(e / n2);
  const int64_t ij = e - iw * n2;
  const int i = (int)(ij / ng), j = (int)(ij % ng);
  const double2 c = chi[e];
  float* xo = x + e * kI;
  xo[0] = (float)qgn[i];
  xo[1] = (float)qgn[j];
  xo[2] = (float)wn[iw];
  xo[3] = (float)(c.x * inv_c);
  xo[4] = (float)(c.y * inv_c);
  if (full && t) {
    const double2 f = full[e];
    t[e * kO] = (float)((f.x - c.x) * inv_c);
    t[e * kO + 1] = (float)((f.y - c.y) * inv_c);
  }
}

__global__ void k_term_apply_dev(double2* __restrict__ chi, const float* __restrict__ y, int ng, int nw,
                                 const double* __restrict__ cs) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t n2 = (int64_t)ng * ng;
  if (e >= n2 * nw) return;
  const double c = cs[0];
  const int iw = (int)(e / n2);
  const int64_t ij = e - iw * n2;
  const int i = (int)(ij / ng), j = (int)(ij % ng);
  const int64_t ji = (int64_t)iw * n2 + (int64_t)j * ng + i;
  const double dre = 0.5 * ((double)y[e * kO] + (double)y[ji * kO]);
  const double dim = 0.5 * ((double)y[e * kO + 1] - (double)y[ji * kO + 1]);
  double2 v = chi[e];
  v.x += c * dre;
  v.y += (i == j) ? 0.0 : c * dim;
  chi[e] = v;
}

// host tables of the feature normalisation for q point iq
void term_tables(chi0_ctx* c, int iq, std::vector<double>& qgn, std::vector<double>& wn) {
  const int ng = c->cfg.ng, nw = c->cfg.nw;
  qgn.resize(ng);
  wn.resize(nw);
  double qmax = 0.0;
  for (int i = 0; i < ng; ++i) {
    double q2 = 0.0;
    for (int d = 0; d < 3; ++d) {
      const double comp = c->q[3 * iq + d] + c->h_gresp[3 * i + d];
      q2 += comp * comp;
    }
    qgn[i] = std::sqrt(q2);
    qmax = std::max(qmax, qgn[i]);
  }
  for (auto& v : qgn) v = qmax > 0 ? v / qmax : 0.0;
  double wmax = 0.0;
  for (int iw = 0; iw < nw; ++iw) wmax = std::max(wmax, std::fabs(c->om[2 * iw + 1]));
  for (int iw = 0; iw < nw; ++iw) wn[iw] = wmax > 0 ? std::fabs(c->om[2 * iw + 1]) / wmax : 0.0;
}

}  // namespace

// tables of the feature normalisation for q point iq (host set-up)
chi0_status term_tables_upload(chi0_ctx* c, int iq) {
  const int ng = c->cfg.ng, nw = c->cfg.nw;
  chi0_status s;
  if ((s = ctx_ensure(c, c->d_termq, (size_t)ng * 8, "terminator tables")) != CHI0_OK) return s;
  if ((s = ctx_ensure(c, c->d_termw, (size_t)nw * 8, "terminator tables")) != CHI0_OK) return s;
  if ((s = ctx_ensure(c, c->d_termc, 16, "terminator scale")) != CHI0_OK) return s;
  std::vector<double> qgn, wn;
  term_tables(c, iq, qgn, wn);
  if (cudaMemcpyAsync(c->d_termq.p, qgn.data(), ng * 8, cudaMemcpyHostToDevice, c->st) != cudaSuccess ||
      cudaMemcpyAsync(c->d_termw.p, wn.data(), nw * 8, cudaMemcpyHostToDevice, c->st) != cudaSuccess ||
      cudaStreamSynchronize(c->st) != cudaSuccess) {
    cudaGetLastError();
    return ctx_fail(c, CHI0_ECUDA, "terminator tables upload failed");
  }
  return CHI0_OK;
}

// kernels: scale c, features (and targets) of chi
chi0_status term_features_launch(chi0_ctx* c, const double2* chi, const double2* full, float* x, float* t) {
  const int ng = c->cfg.ng, nw = c->cfg.nw;
  k_diag_scale<<<1, 256, 0, c->st>>>(chi, ng, (double*)c->d_termc.p);
  const int64_t n = (int64_t)ng * ng * nw;
  k_term_features_dev<<<(unsigned)((n + 255) / 256), 256, 0, c->st>>>(
      chi, full, (const double*)c->d_termq.p, (const double*)c->d_termw.p, ng, nw,
      (const double*)c->d_termc.p, x, t);
  if (cudaGetLastError() != cudaSuccess) return ctx_fail(c, CHI0_ECUDA, "terminator features launch failed");
  return CHI0_OK;
}

chi0_status term_plan(chi0_ctx* c, int iq) {
  const int64_t n = (int64_t)c->cfg.ng * c->cfg.ng * c->cfg.nw;
  chi0_status s;
  if ((s = ctx_ensure(c, c->d_termx, (size_t)n * kI * 4, "terminator features")) != CHI0_OK) return s;
  if ((s = ctx_ensure(c, c->d_termy, (size_t)n * kO * 4, "terminator prediction")) != CHI0_OK) return s;
  return term_tables_upload(c, iq);
}

// chi += Hermitised network correction (build_chi0 with a terminator set)
chi0_status term_launch(chi0_ctx* c, double2* chi) {
  const int ng = c->cfg.ng, nw = c->cfg.nw;
  const int64_t n = (int64_t)ng * ng * nw;
  chi0_status s;
  if ((s = term_features_launch(c, chi, nullptr, (float*)c->d_termx.p, nullptr)) != CHI0_OK) return s;
  if (mlp_predict(c->term_params, (const float*)c->d_termx.p, n, c->term_bf16, (float*)c->d_termy.p,
                  c->st) != cudaSuccess) {
    cudaGetLastError();
    return ctx_fail(c, CHI0_ECUDA, "terminator prediction launch failed");
  }
  k_term_apply_dev<<<(unsigned)((n + 255) / 256), 256, 0, c->st>>>(chi, (const float*)c->d_termy.p, ng, nw,
                                                                   (const double*)c->d_termc.p);
  if (cudaGetLastError() != cudaSuccess) return ctx_fail(c, CHI0_ECUDA, "terminator apply launch failed");
  c->launches += 4;
  return CHI0_OK;
}

}  // namespace chi0

extern "C" {

int chi0_mlp_nparams(void) { return chi0::kP; }

int64_t chi0_mlp_workspace_floats(int64_t batch) {
  const int64_t nblk = (batch + chi0::kS - 1) / chi0::kS;
  return nblk * chi0::kP + nblk;
}

chi0_status chi0_mlp_loss_grad(const float* params, const float* x, const float* t, int64_t batch,
                               int bf16, float* grad, float* loss, float* work, void* stream) {
  if (!params || !x || !t || !grad || !work || batch < 1) return CHI0_EINVAL;
  const int64_t nblk = (batch + chi0::kS - 1) / chi0::kS;
  if (nblk > 0x7fffffff) return CHI0_EINVAL;
  if (chi0::mlp_loss_grad(params, x, t, batch, bf16, grad, loss, work, work + nblk * chi0::kP,
                          (cudaStream_t)stream) != cudaSuccess) {
    cudaGetLastError();
    return CHI0_ECUDA;
  }
  return CHI0_OK;
}

chi0_status chi0_mlp_adam(float* params, const float* grad, float* m, float* v, int64_t n, float lr,
                          float beta1, float beta2, float eps, int step, void* stream) {
  if (!params || !grad || !m || !v || n < 1 || step < 1) return CHI0_EINVAL;
  if (chi0::mlp_adam(params, grad, m, v, n, lr, beta1, beta2, eps, step, (cudaStream_t)stream) != cudaSuccess) {
    cudaGetLastError();
    return CHI0_ECUDA;
  }
  return CHI0_OK;
}

chi0_status chi0_mlp_predict(const float* params, const float* x, int64_t batch, int bf16, float* y,
                             void* stream) {
  if (!params || !x || !y || batch < 1) return CHI0_EINVAL;
  if (chi0::mlp_predict(params, x, batch, bf16, y, (cudaStream_t)stream) != cudaSuccess) {
    cudaGetLastError();
    return CHI0_ECUDA;
  }
  return CHI0_OK;
}

chi0_status chi0_term_features(chi0_ctx* c, int iq, const void* chi_trunc, const void* chi_full, float* x,
                               float* t, double* scale) {
  if (!c) return CHI0_EINVAL;
  if (iq < 0 || iq >= c->cfg.nq || !chi_trunc || !x || (chi_full && !t))
    return chi0::ctx_fail(c, CHI0_EINVAL, "bad iq or NULL buffer");
  if (c->h_gresp.empty() || c->rho_iq != iq)
    return chi0::ctx_fail(c, CHI0_ESTATE, "chi0_compute_rho(iq) must come first (response G set)");
  chi0_status s = chi0::term_tables_upload(c, iq);
  if (s != CHI0_OK) return s;
  s = chi0::term_features_launch(c, (const double2*)chi_trunc, (const double2*)chi_full, x, t);
  if (s != CHI0_OK) return s;
  if (scale) {
    double cs[2];
    if (cudaMemcpyAsync(cs, c->d_termc.p, 16, cudaMemcpyDeviceToHost, c->st) != cudaSuccess ||
        cudaStreamSynchronize(c->st) != cudaSuccess) {
      cudaGetLastError();
      return chi0::ctx_fail(c, CHI0_ECUDA, "scale read back failed");
    }
    *scale = cs[0];
  }
  return CHI0_OK;
}

chi0_status chi0_set_terminator(chi0_ctx* c, const float* params, int bf16) {
  if (!c) return CHI0_EINVAL;
  if (params && c->bg_on)
    return chi0::ctx_fail(c, CHI0_EINVAL, "the extrapolar terminator is set: the two corrections exclude each other");
  c->term_params = params;
  c->term_bf16 = bf16;
  c->chi_iq = c->eps_iq = -1;
  ++c->plan_epoch;
  return CHI0_OK;
}

}  // extern "C"
