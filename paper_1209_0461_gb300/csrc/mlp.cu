// Learned response surrogate: a 3-layer perceptron (n_in -> 128 -> 128 -> 1,
// tanh) with BF16 weight matrices, FP32 biases and FP32 accumulation, and its
// training kernels (mean-squared-error gradient by the chain rule, Adam).  It
// maps per-bin features of a kick to ln R_b (R_b = P_nu^{1/2} / P_cdm^{1/2} of
// Eq. P-final); the paper has no learned part.
//
// Layout of the flat parameter vector (FP32 master copy):
//   W1 [128][n_in], b1 [128], W2 [128][128], b2 [128], w3 [128], b3 [1]
//
// Kernels:
//   k_mlp_forward   y = y_mu + y_sigma * out(x): a warp per 16 samples, layer 2
//                   on the tensor cores from activations split in three BF16
//   k_mlp_backward  per-CTA partial gradients and loss, fixed tile order; one CTA
//                   of 256 threads per SM, tiles of 32 samples, register tiles of
//                   two hidden units x eight samples (FP32)
//   k_mlp_reduce    sum of the CTA partials in a fixed order (deterministic)
//   k_mlp_adam      Adam on the master copy, then the BF16 weight copies
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include <new>
#include <vector>

#include "nupm_internal.h"

namespace nupm {
namespace {

constexpr int kW = 128;        // hidden width
constexpr int kMaxIn = 16;     // input features (<=)
constexpr int kTS = 32;        // samples per tile of the backward pass
constexpr int kHP = 36;        // padded row of the [unit][sample] tiles (16-byte rows)
constexpr int kWP = 129;       // padded row of the 128x128 shared matrix
constexpr int kBwdThreads = 256;

// Shared-memory layout (floats) of the backward kernel.
struct MlpSmem {
  static constexpr int W2 = 0;                        // W2s[k][j] = W2[j][k], rows of kWP
  static constexpr int H1 = W2 + kW * kWP;             // h1T[k][s], rows of kHP
  static constexpr int DZ2 = H1 + kW * kHP;            // dz2T[j][s]
  static constexpr int XH = DZ2 + kW * kHP;            // xh[s][i], rows of kMaxIn
  static constexpr int OUT = XH + kTS * kMaxIn;        // squared residuals
  static constexpr int DOUT = OUT + kTS;               // dL/dout per sample
  static constexpr int RED = DOUT + kTS;               // [8 warps][8 samples] reduction
  static constexpr int TOTAL = RED + 64;
  static constexpr size_t BYTES = (size_t)TOTAL * sizeof(float);
  static_assert(H1 % 4 == 0 && XH % 4 == 0, "16-byte rows");
  static_assert(4 * kW * (kMaxIn + 3) <= TOTAL - H1, "the end sums reuse what follows W2");
};

// Shared memory of the forward kernel: W2 as B fragments of m16n8k16
// [k tile][n tile][lane] (8 bytes), W1 rows of kW1P floats, b1, (b2, w3) pairs
// per unit, one staging tile of 16 x kXP inputs per warp.
constexpr int kFwdWarps = 4;
constexpr int kW1P = 20;       // rows of two units apart by 40 words: the quads' 16-byte reads miss each other's banks
constexpr int kXP = 20;
struct FwdSmem {
  static constexpr int B = 0;
  static constexpr int W1 = B + kW * kW * 2;
  static constexpr int B1 = W1 + kW * kW1P * 4;
  static constexpr int BW = B1 + kW * 4;
  static constexpr int X = BW + kW * 8;
  static constexpr int BYTES = X + kFwdWarps * 16 * kXP * 4;
};

struct MlpArgs {
  int n_in;
  int64_t n;                          // samples
  const float* X;                     // [n][n_in] raw features
  const float* Y;                     // [n] raw targets (ln R), backward only
  float* out;                         // [n] forward output (ln R)
  const __nv_bfloat16* W1;            // [128][n_in]
  const float* b1;
  const __nv_bfloat16* W2;            // [128][128]
  const float* b2;
  const __nv_bfloat16* w3;            // [128]
  const float* b3;
  const float* mu;                    // [n_in]
  const float* sig;                   // [n_in]
  float y_mu, y_sig;
  float* partial;                     // [gridDim][P + 1] (backward)
  int64_t P;                          // parameter count
};

__device__ __forceinline__ float bf(__nv_bfloat16 v) { return __bfloat162float(v); }

// h = hi + mid + lo to 2^-27 relative, each a BF16 (products with the BF16
// weights are then exact); two neighbouring values packed per word.
__device__ __forceinline__ void split3(float x, float y, uint32_t (&w)[3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(x, y);
    w[i] = *reinterpret_cast<const uint32_t*>(&p);
    x -= __low2float(p);
    y -= __high2float(p);
  }
}

__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t a0, const uint32_t a1, const uint32_t a2,
                                         const uint32_t a3, uint2 b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b.x), "r"(b.y));
}

// Two packed BF16 values with those that are not finite replaced by zero.
__device__ __forceinline__ uint32_t finite_part(uint32_t w) {
  const uint32_t lo = (w & 0x7f80u) == 0x7f80u ? 0u : 0xffffu;
  const uint32_t hi = (w & 0x7f800000u) == 0x7f800000u ? 0u : 0xffff0000u;
  return w & (lo | hi);
}

// One warp per 16 samples.  Lane (g, q) = (lane / 4, lane % 4) holds rows g and
// g + 8; layer 1 is evaluated straight into the A fragments of layer 2: per k
// tile of 16 hidden units the lane needs units 2q, 2q + 1, 2q + 8, 2q + 9 of
// its two rows.  Layer 2, 128 x 128 with BF16 weights, runs on the tensor
// cores with h1 as three BF16 words, so no activation is rounded; each k tile's
// product starts from zero (low word first) and is added to the FP32 sum in
// round-to-nearest, because the tensor cores' own accumulation truncates.
// The warp-level mma is taken rather than a tcgen05 tile: what bounds the kernel is
// the 256 tanh and the FP32 work of a sample, and the fragments stay in
// registers between the layers.  500k samples take 0.248 ms (74 TFLOP/s; error
// against 64 bits 4.8e-8); one CTA of 128 threads per SM, each thread a hidden
// unit of 32 samples in FP32, took 1.07 ms (four warps per SM; 5.6e-8).
__global__ void __launch_bounds__(kFwdWarps * 32, 3) k_mlp_forward(MlpArgs A) {
  extern __shared__ __align__(16) unsigned char smf[];
  uint2* Bs = reinterpret_cast<uint2*>(smf + FwdSmem::B);
  float* W1s = reinterpret_cast<float*>(smf + FwdSmem::W1);
  float* b1s = reinterpret_cast<float*>(smf + FwdSmem::B1);
  float2* bw = reinterpret_cast<float2*>(smf + FwdSmem::BW);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, q = lane & 3;
  float* xs = reinterpret_cast<float*>(smf + FwdSmem::X) + warp * 16 * kXP;
  // fragment (kt, nt, lane): W2[8 nt + g][16 kt + 2q + {0, 1}] and + 8; weights that
  // are not finite apart (below)
  uint32_t apart = 0;
  for (int i = threadIdx.x; i < 8 * 16 * 32; i += blockDim.x) {
    const int l = i & 31, nt = (i >> 5) & 15, kt = i >> 9;
    const __nv_bfloat16* w = A.W2 + (8 * nt + (l >> 2)) * kW + 16 * kt + 2 * (l & 3);
    const uint2 b = make_uint2(*reinterpret_cast<const uint32_t*>(w), *reinterpret_cast<const uint32_t*>(w + 8));
    const uint2 f = make_uint2(finite_part(b.x), finite_part(b.y));
    Bs[i] = f;
    apart |= (f.x ^ b.x) | (f.y ^ b.y);
  }
  for (int i = threadIdx.x; i < kW * kMaxIn; i += blockDim.x) {
    const int u = i / kMaxIn, c = i % kMaxIn;
    W1s[u * kW1P + c] = c < A.n_in ? bf(A.W1[u * A.n_in + c]) : 0.0f;
  }
  for (int i = threadIdx.x; i < kW; i += blockDim.x) {
    b1s[i] = A.b1[i];
    bw[i] = make_float2(A.b2[i], bf(A.w3[i]));
  }
  const bool odd = __syncthreads_or(apart != 0);
  // units u, u + 1 of layer 1 for two rows of inputs: h[row][unit]
  auto layer1 = [&](const float (&x)[2][kMaxIn], int u, float (&h)[2][2]) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      float acc0 = b1s[u + e], acc1 = acc0;
#pragma unroll
      for (int c = 0; c < kMaxIn; c += 4) {
        const float4 w = *reinterpret_cast<const float4*>(W1s + (u + e) * kW1P + c);
        acc0 = fmaf(w.x, x[0][c], acc0);
        acc1 = fmaf(w.x, x[1][c], acc1);
        acc0 = fmaf(w.y, x[0][c + 1], acc0);
        acc1 = fmaf(w.y, x[1][c + 1], acc1);
        acc0 = fmaf(w.z, x[0][c + 2], acc0);
        acc1 = fmaf(w.z, x[1][c + 2], acc1);
        acc0 = fmaf(w.w, x[0][c + 3], acc0);
        acc1 = fmaf(w.w, x[1][c + 3], acc1);
      }
      h[0][e] = tanhf(acc0);
      h[1][e] = tanhf(acc1);
    }
  };
  const float b3 = A.b3[0];
  const int64_t tiles = (A.n + 15) / 16;
  for (int64_t t = (int64_t)blockIdx.x * kFwdWarps + warp; t < tiles; t += (int64_t)gridDim.x * kFwdWarps) {
    const int64_t s0 = t * 16;
    __syncwarp();
    for (int i = lane; i < 16 * kMaxIn; i += 32) {   // unused columns and rows past n: 0
      const int r = i / kMaxIn, c = i % kMaxIn;
      const int64_t row = s0 + r;
      xs[r * kXP + c] = (c < A.n_in && row < A.n) ? (A.X[row * A.n_in + c] - A.mu[c]) / A.sig[c] : 0.0f;
    }
    __syncwarp();
    float x[2][kMaxIn];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int c = 0; c < kMaxIn; c += 4) {
        const float4 v = *reinterpret_cast<const float4*>(xs + (g + 8 * r) * kXP + c);
        x[r][c] = v.x;
        x[r][c + 1] = v.y;
        x[r][c + 2] = v.z;
        x[r][c + 3] = v.w;
      }
    float z[16][4];
#pragma unroll
    for (int nt = 0; nt < 16; ++nt) z[nt][0] = z[nt][1] = z[nt][2] = z[nt][3] = 0.0f;
    // Weights that are not finite (a master weight past the BF16 range is one): times
    // the high word of h1 alone, which has its sign.  The lower words may be zero or of
    // the other sign, and their product or the sum would be a NaN.
    if (odd) {
#pragma unroll 1
      for (int kt = 0; kt < 8; ++kt) {
        uint32_t a[4];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
          float h[2][2];
          layer1(x, 16 * kt + 8 * p + 2 * q, h);
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            const __nv_bfloat162 v = __floats2bfloat162_rn(h[r][0], h[r][1]);
            a[2 * p + r] = *reinterpret_cast<const uint32_t*>(&v);
          }
        }
#pragma unroll
        for (int nt = 0; nt < 16; ++nt) {
          const __nv_bfloat16* w = A.W2 + (8 * nt + g) * kW + 16 * kt + 2 * q;
          const uint2 b = make_uint2(*reinterpret_cast<const uint32_t*>(w), *reinterpret_cast<const uint32_t*>(w + 8));
          mma_bf16(z[nt], a[0], a[1], a[2], a[3], make_uint2(b.x ^ finite_part(b.x), b.y ^ finite_part(b.y)));
        }
      }
    }
#pragma unroll 1
    for (int kt = 0; kt < 8; ++kt) {
      uint32_t a[4][3];   // [fragment word][hi, mid, lo]
#pragma unroll
      for (int p = 0; p < 2; ++p) {   // units 16 kt + 8 p + 2 q + {0, 1}
        float h[2][2];                // [row][unit]
        layer1(x, 16 * kt + 8 * p + 2 * q, h);
        split3(h[0][0], h[0][1], a[2 * p]);
        split3(h[1][0], h[1][1], a[2 * p + 1]);
      }
      const uint2* bk = Bs + kt * 16 * 32 + lane;
#pragma unroll
      for (int nt = 0; nt < 16; ++nt) {
        const uint2 b = bk[nt * 32];
        float c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        mma_bf16(c, a[0][2], a[1][2], a[2][2], a[3][2], b);
        mma_bf16(c, a[0][1], a[1][1], a[2][1], a[3][1], b);
        mma_bf16(c, a[0][0], a[1][0], a[2][0], a[3][0], b);
#pragma unroll
        for (int e = 0; e < 4; ++e) z[nt][e] += c[e];
      }
    }
    // layer 3 over the lane's 32 columns, then over the four lanes of the row
    float o0 = 0.0f, o1 = 0.0f;
#pragma unroll
    for (int nt = 0; nt < 16; ++nt)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float2 w = bw[8 * nt + 2 * q + e];
        o0 = fmaf(w.y, tanhf(z[nt][e] + w.x), o0);
        o1 = fmaf(w.y, tanhf(z[nt][2 + e] + w.x), o1);
      }
#pragma unroll
    for (int m = 1; m < 4; m <<= 1) {
      o0 += __shfl_xor_sync(0xffffffffu, o0, m);
      o1 += __shfl_xor_sync(0xffffffffu, o1, m);
    }
    if (q == 0) {
      if (s0 + g < A.n) A.out[s0 + g] = A.y_mu + A.y_sig * (o0 + b3);
      if (s0 + g + 8 < A.n) A.out[s0 + g + 8] = A.y_mu + A.y_sig * (o1 + b3);
    }
  }
}

// Partial gradient of L = (1/n) sum (out - (Y - y_mu)/y_sig)^2 over the tiles
// blockIdx.x, blockIdx.x + gridDim.x, ... (in that order), written to
// partial[blockIdx.x][0..P) in the flat parameter layout, the partial loss
// at [P].  Thread (jj, sg) = (tid % 64, tid / 64) owns hidden units jj and
// jj + 64 for the samples 8 sg .. 8 sg + 7 (layers 1 and 2 and their
// gradients: 16 multiply-adds for two scalar and two 16-byte shared reads) and, for dW2, the
// same two units against k = 32 sg .. 32 sg + 31 over all samples, kept in 64
// registers across tiles.  29 us for 4096 samples; one CTA of 128 threads with
// dW2 in shared memory, four warps per SM, took 48 us.
__global__ void __launch_bounds__(kBwdThreads, 1) k_mlp_backward(MlpArgs A) {
  extern __shared__ __align__(16) float sm[];
  const int tid = threadIdx.x, jj = tid & 63, sg = tid >> 6, lane = tid & 31, warp = tid >> 5;
  const int ju[2] = {jj, jj + 64};
  float* W2s = sm + MlpSmem::W2;
  float* h1T = sm + MlpSmem::H1;
  float* dz2T = sm + MlpSmem::DZ2;
  float* xh = sm + MlpSmem::XH;
  float* outs = sm + MlpSmem::OUT;
  float* dout = sm + MlpSmem::DOUT;
  float* red = sm + MlpSmem::RED;
  // W2, eight BF16 a load and all of a thread's loads in flight (2-byte loads took
  // sixteen round trips, 2 us of a minibatch that is one tile a CTA)
  uint4 wv[kW * kW / 8 / kBwdThreads];
#pragma unroll
  for (int q = 0; q < kW * kW / 8 / kBwdThreads; ++q) wv[q] = reinterpret_cast<const uint4*>(A.W2)[tid + q * kBwdThreads];
#pragma unroll
  for (int q = 0; q < kW * kW / 8 / kBwdThreads; ++q) {
    const int idx = 8 * (tid + q * kBwdThreads), j = idx / kW, k = idx % kW;   // W2[j][k .. k + 7]
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&wv[q]);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      W2s[(k + 2 * e) * kWP + j] = __low2float(h[e]);
      W2s[(k + 2 * e + 1) * kWP + j] = __high2float(h[e]);
    }
  }
  float dW2[2][32], dW1[2][kMaxIn], db1[2] = {0.0f, 0.0f}, db2[2] = {0.0f, 0.0f}, dw3[2] = {0.0f, 0.0f};
  float db3 = 0.0f, loss = 0.0f, w3[2], b1[2], b2[2];
#pragma unroll
  for (int e = 0; e < 2; ++e) {
#pragma unroll
    for (int k = 0; k < 32; ++k) dW2[e][k] = 0.0f;
#pragma unroll
    for (int i = 0; i < kMaxIn; ++i) dW1[e][i] = 0.0f;
    w3[e] = bf(A.w3[ju[e]]);
    b1[e] = A.b1[ju[e]];
    b2[e] = A.b2[ju[e]];
  }
  const float inv_n = 1.0f / (float)A.n, b3 = A.b3[0];
  const int64_t tiles = (A.n + kTS - 1) / kTS;
  for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const int64_t s0 = t * kTS;
    for (int idx = tid; idx < kTS * kMaxIn; idx += kBwdThreads) {   // unused columns and rows past n: 0
      const int s = idx / kMaxIn, i = idx % kMaxIn;
      const int64_t row = s0 + s;
      xh[idx] = (i < A.n_in && row < A.n) ? (A.X[row * A.n_in + i] - A.mu[i]) / A.sig[i] : 0.0f;
    }
    __syncthreads();
    // layer 1
    float h1[2][8];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      float w[kMaxIn];
#pragma unroll
      for (int i = 0; i < kMaxIn; ++i) w[i] = i < A.n_in ? bf(A.W1[ju[e] * A.n_in + i]) : 0.0f;
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        float acc = b1[e];
#pragma unroll
        for (int i = 0; i < kMaxIn; ++i) acc = fmaf(w[i], xh[(8 * sg + s) * kMaxIn + i], acc);
        h1[e][s] = tanhf(acc);
      }
      float4* d = reinterpret_cast<float4*>(h1T + ju[e] * kHP + 8 * sg);
      d[0] = make_float4(h1[e][0], h1[e][1], h1[e][2], h1[e][3]);
      d[1] = make_float4(h1[e][4], h1[e][5], h1[e][6], h1[e][7]);
    }
    __syncthreads();
    // layer 2: h2[s] = tanh(b2[j] + sum_k W2[j][k] h1[s][k])
    float h2[2][8];
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
      for (int s = 0; s < 8; ++s) h2[e][s] = b2[e];
#pragma unroll 4
    for (int k = 0; k < kW; ++k) {
      const float wa = W2s[k * kWP + jj], wb = W2s[k * kWP + jj + 64];
      const float4* hk = reinterpret_cast<const float4*>(h1T + k * kHP + 8 * sg);
      const float4 u = hk[0], v = hk[1];
      const float hv[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        h2[0][s] = fmaf(wa, hv[s], h2[0][s]);
        h2[1][s] = fmaf(wb, hv[s], h2[1][s]);
      }
    }
    // layer 3: out[s] = b3 + sum_j w3[j] h2[s][j], fixed reduction tree
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      h2[0][s] = tanhf(h2[0][s]);
      h2[1][s] = tanhf(h2[1][s]);
      float v = fmaf(w3[0], h2[0][s], w3[1] * h2[1][s]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) red[warp * 8 + s] = v;
    }
    __syncthreads();
    // dL/dout per sample (zero past n)
    if (tid < kTS) {
      const int64_t row = s0 + tid;
      const int w0 = 2 * (tid >> 3) * 8 + (tid & 7);
      float d = 0.0f, r2 = 0.0f;
      if (row < A.n) {
        const float r = b3 + (red[w0] + red[w0 + 8]) - (A.Y[row] - A.y_mu) / A.y_sig;
        d = 2.0f * r * inv_n;
        r2 = r * r;
      }
      dout[tid] = d;
      outs[tid] = r2;
    }
    __syncthreads();
    if (tid == 0)
      for (int s = 0; s < kTS; ++s) {
        loss += outs[s];
        db3 += dout[s];
      }
    // the pre-activation gradient of layer 2
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      float dz[8];
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        const float d = dout[8 * sg + s];
        dw3[e] = fmaf(d, h2[e][s], dw3[e]);
        dz[s] = d * w3[e] * (1.0f - h2[e][s] * h2[e][s]);
        db2[e] += dz[s];
      }
      float4* p = reinterpret_cast<float4*>(dz2T + ju[e] * kHP + 8 * sg);
      p[0] = make_float4(dz[0], dz[1], dz[2], dz[3]);
      p[1] = make_float4(dz[4], dz[5], dz[6], dz[7]);
    }
    __syncthreads();
    // dW2[j][k] += sum_s dz2[s] h1[s][k], k = 32 sg + kk
#pragma unroll 1
    for (int s4 = 0; s4 < kTS / 4; ++s4) {
      const float4 da = *reinterpret_cast<const float4*>(dz2T + jj * kHP + 4 * s4);
      const float4 db = *reinterpret_cast<const float4*>(dz2T + (jj + 64) * kHP + 4 * s4);
      const float* hb = h1T + 32 * sg * kHP + 4 * s4;
#pragma unroll
      for (int kk = 0; kk < 32; ++kk) {
        const float4 h = *reinterpret_cast<const float4*>(hb + kk * kHP);
        dW2[0][kk] = fmaf(da.x, h.x, dW2[0][kk]);
        dW2[1][kk] = fmaf(db.x, h.x, dW2[1][kk]);
        dW2[0][kk] = fmaf(da.y, h.y, dW2[0][kk]);
        dW2[1][kk] = fmaf(db.y, h.y, dW2[1][kk]);
        dW2[0][kk] = fmaf(da.z, h.z, dW2[0][kk]);
        dW2[1][kk] = fmaf(db.z, h.z, dW2[1][kk]);
        dW2[0][kk] = fmaf(da.w, h.w, dW2[0][kk]);
        dW2[1][kk] = fmaf(db.w, h.w, dW2[1][kk]);
      }
    }
    // layer-1 units k = jj, jj + 64: dh1[s] = sum_j W2[j][k] dz2[s][j]
    float dh[2][8];
#pragma unroll
    for (int s = 0; s < 8; ++s) dh[0][s] = dh[1][s] = 0.0f;
#pragma unroll 4
    for (int j = 0; j < kW; ++j) {
      const float wa = W2s[jj * kWP + j], wb = W2s[(jj + 64) * kWP + j];
      const float4* dz = reinterpret_cast<const float4*>(dz2T + j * kHP + 8 * sg);
      const float4 u = dz[0], v = dz[1];
      const float dv[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        dh[0][s] = fmaf(wa, dv[s], dh[0][s]);
        dh[1][s] = fmaf(wb, dv[s], dh[1][s]);
      }
    }
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const float* xr = xh + (8 * sg + s) * kMaxIn;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float dz1 = dh[e][s] * (1.0f - h1[e][s] * h1[e][s]);
        db1[e] += dz1;
#pragma unroll
        for (int i = 0; i < kMaxIn; ++i) dW1[e][i] = fmaf(dz1, xr[i], dW1[e][i]);
      }
    }
    __syncthreads();   // h1T, dz2T, xh and outs are rewritten by the next tile
  }
  // write this CTA's partials in the flat layout; the four sample groups' sums
  // of W1, b1, b2 and w3 are added in group order
  float* out = A.partial + (int64_t)blockIdx.x * (A.P + 1);
  const int n_in = A.n_in;
  const int oW1 = 0, ob1 = kW * n_in, oW2 = ob1 + kW, ob2 = oW2 + kW * kW, ow3 = ob2 + kW, ob3 = ow3 + kW;
  constexpr int NS = kMaxIn + 3;
  float* ends = sm + MlpSmem::H1;                       // [4][NS][kW]
#pragma unroll
  for (int e = 0; e < 2; ++e) {
#pragma unroll
    for (int k = 0; k < 32; ++k) W2s[ju[e] * kWP + 32 * sg + k] = dW2[e][k];   // for whole-row stores
    float* d = ends + sg * NS * kW + ju[e];
#pragma unroll
    for (int i = 0; i < kMaxIn; ++i) d[i * kW] = dW1[e][i];
    d[kMaxIn * kW] = db1[e];
    d[(kMaxIn + 1) * kW] = db2[e];
    d[(kMaxIn + 2) * kW] = dw3[e];
  }
  __syncthreads();
  for (int idx = tid; idx < kW * kW; idx += kBwdThreads) out[oW2 + idx] = W2s[(idx / kW) * kWP + idx % kW];
  for (int idx = tid; idx < NS * kW; idx += kBwdThreads) {
    const int i = idx / kW, j = idx % kW;
    if (i < kMaxIn && i >= n_in) continue;
    float v = 0.0f;
#pragma unroll
    for (int q = 0; q < 4; ++q) v += ends[q * NS * kW + idx];
    const int o = i < kMaxIn ? oW1 + j * n_in + i : i == kMaxIn ? ob1 + j : i == kMaxIn + 1 ? ob2 + j : ow3 + j;
    out[o] = v;
  }
  if (tid == 0) {
    out[ob3] = db3;
    out[A.P] = loss * inv_n;
  }
}

// grad[p] = sum over the CTA partials, loss = the same sum at index P; either
// may be null.  A CTA takes 32 parameters: warp w adds rows w, w + 8, ..., then one warp
// adds the eight in order: 4.5 us for 128 rows (one thread a parameter adding
// the rows one after another took 14 us).
constexpr int kRedWarps = 8;
__global__ void __launch_bounds__(kRedWarps * 32) k_mlp_reduce(const float* __restrict__ partial, int nblk,
                                                             int64_t P, float* __restrict__ grad,
                                                             float* __restrict__ loss) {
  __shared__ float red[kRedWarps][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t p = (int64_t)blockIdx.x * 32 + lane;
  float acc = 0.0f;
  if (p <= P) {
#pragma unroll 8
    for (int b = warp; b < nblk; b += kRedWarps) acc += partial[(int64_t)b * (P + 1) + p];
  }
  red[warp][lane] = acc;
  __syncthreads();
  if (warp == 0 && p <= P) {
    float v = 0.0f;
#pragma unroll
    for (int w = 0; w < kRedWarps; ++w) v += red[w][lane];
    if (p < P) {
      if (grad) grad[p] = v;
    } else if (loss) {
      *loss = v;
    }
  }
}

// Adam (Kingma & Ba 2015) on the FP32 master copy, then the BF16 copies of
// the weight matrices.  bc1 = 1 - beta1^t, bc2 = 1 - beta2^t.
__global__ void k_mlp_adam(float* __restrict__ theta, const float* __restrict__ g, float* __restrict__ m,
                           float* __restrict__ v, int64_t P, float lr, float b1, float b2, float eps, float bc1,
                           float bc2, __nv_bfloat16* __restrict__ wbf, int n_in) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= P) return;
  const float gp = g[p];
  const float mp = b1 * m[p] + (1.0f - b1) * gp;
  const float vp = b2 * v[p] + (1.0f - b2) * gp * gp;
  m[p] = mp;
  v[p] = vp;
  const float th = theta[p] - lr * (mp / bc1) / (sqrtf(vp / bc2) + eps);
  theta[p] = th;
  const int64_t ob1 = (int64_t)kW * n_in, oW2 = ob1 + kW, ob2 = oW2 + (int64_t)kW * kW, ow3 = ob2 + kW;
  if (p < ob1) wbf[p] = __float2bfloat16_rn(th);                                // W1
  else if (p >= oW2 && p < ob2) wbf[ob1 + (p - oW2)] = __float2bfloat16_rn(th);   // W2
  else if (p >= ow3 && p < ow3 + kW) wbf[ob1 + kW * kW + (p - ow3)] = __float2bfloat16_rn(th);   // w3
}

// BF16 copies of the weight matrices from the master copy.
__global__ void k_mlp_to_bf16(const float* __restrict__ theta, __nv_bfloat16* __restrict__ wbf, int n_in) {
  const int64_t ob1 = (int64_t)kW * n_in, oW2 = ob1 + kW, ob2 = oW2 + (int64_t)kW * kW, ow3 = ob2 + kW;
  const int64_t nb = ob1 + (int64_t)kW * kW + kW;
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nb) return;
  int64_t p;
  if (q < ob1) p = q;
  else if (q < ob1 + kW * kW) p = oW2 + (q - ob1);
  else p = ow3 + (q - ob1 - kW * kW);
  wbf[q] = __float2bfloat16_rn(theta[p]);
}

}  // namespace
}  // namespace nupm

using namespace nupm;

struct pm_mlp {
  int n_in = 0;
  int64_t P = 0;
  cudaStream_t stream = nullptr;
  int sm_count = 152;
  float* theta = nullptr;          // [P] master
  float* m = nullptr;
  float* v = nullptr;
  float* grad = nullptr;           // [P]
  float* partial = nullptr;        // [nblk][P + 1]
  __nv_bfloat16* wbf = nullptr;    // W1 | W2 | w3
  float* norm = nullptr;           // mu [n_in] | sigma [n_in]
  float y_mu = 0.0f, y_sig = 1.0f;
  int64_t step = 0;
  int nblk = 0;
};

namespace {

int mlp_check(cudaError_t e) { return e == cudaSuccess ? PM_OK : PM_ERR_CUDA; }

MlpArgs mlp_args(const pm_mlp* m, const float* X, const float* Y, int64_t n, float* out) {
  MlpArgs A{};
  A.n_in = m->n_in;
  A.n = n;
  A.X = X;
  A.Y = Y;
  A.out = out;
  A.W1 = m->wbf;
  A.b1 = m->theta + (int64_t)kW * m->n_in;
  A.W2 = m->wbf + (int64_t)kW * m->n_in;
  A.b2 = m->theta + (int64_t)kW * m->n_in + kW + (int64_t)kW * kW;
  A.w3 = m->wbf + (int64_t)kW * m->n_in + (int64_t)kW * kW;
  A.b3 = m->theta + m->P - 1;
  A.mu = m->norm;
  A.sig = m->norm + m->n_in;
  A.y_mu = m->y_mu;
  A.y_sig = m->y_sig;
  A.partial = m->partial;
  A.P = m->P;
  return A;
}

// Gradient and loss of a batch into DEVICE grad [P] and loss [1] (either may be null).
int mlp_grad_launch(pm_mlp* m, const float* X, const float* Y, int64_t n, float* grad, float* loss) {
  MlpArgs A = mlp_args(m, X, Y, n, nullptr);
  const int64_t tiles = (n + kTS - 1) / kTS;
  const int grid = (int)(tiles < m->nblk ? tiles : m->nblk);
  k_mlp_backward<<<grid, kBwdThreads, MlpSmem::BYTES, m->stream>>>(A);
  k_mlp_reduce<<<(unsigned)((m->P + 1 + 31) / 32), kRedWarps * 32, 0, m->stream>>>(m->partial, grid, m->P, grad, loss);
  return mlp_check(cudaGetLastError());
}

}  // namespace

namespace nupm {

int mlp_inputs(const pm_mlp* m) { return m ? m->n_in : 0; }

int mlp_forward_on(pm_mlp* m, const float* X, int64_t n, float* y, cudaStream_t s) {
  if (!m || n < 0 || (n > 0 && (!X || !y))) return PM_ERR_INVALID;
  if (n == 0) return PM_OK;
  MlpArgs A = mlp_args(m, X, nullptr, n, y);
  const int64_t ctas = ((n + 15) / 16 + kFwdWarps - 1) / kFwdWarps;
  const int grid = (int)(ctas < 3 * m->sm_count ? ctas : 3 * m->sm_count);
  k_mlp_forward<<<grid, kFwdWarps * 32, FwdSmem::BYTES, s>>>(A);
  return mlp_check(cudaGetLastError());
}

}  // namespace nupm

extern "C" {

int pm_mlp_create(int32_t n_in, int32_t width, void* cuda_stream, pm_mlp** out) {
  if (!out) return PM_ERR_INVALID;
  *out = nullptr;
  if (n_in < 1 || n_in > kMaxIn || width != kW) return PM_ERR_INVALID;
  pm_mlp* m = new (std::nothrow) pm_mlp;
  if (!m) return PM_ERR_ALLOC;
  m->n_in = n_in;
  m->P = (int64_t)kW * n_in + kW + (int64_t)kW * kW + kW + kW + 1;
  m->stream = static_cast<cudaStream_t>(cuda_stream);
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&m->sm_count, cudaDevAttrMultiProcessorCount, dev);
  m->nblk = m->sm_count;
  const size_t pb = (size_t)m->P * sizeof(float);
  bool ok = cudaMalloc(&m->theta, pb) == cudaSuccess && cudaMalloc(&m->m, pb) == cudaSuccess &&
            cudaMalloc(&m->v, pb) == cudaSuccess && cudaMalloc(&m->grad, pb + sizeof(float)) == cudaSuccess &&
            cudaMalloc(&m->partial, (size_t)m->nblk * (m->P + 1) * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&m->wbf, (size_t)((int64_t)kW * n_in + (int64_t)kW * kW + kW) * sizeof(__nv_bfloat16)) ==
                cudaSuccess &&
            cudaMalloc(&m->norm, 2 * (size_t)n_in * sizeof(float)) == cudaSuccess;
  if (ok) {
    ok = cudaMemsetAsync(m->theta, 0, pb, m->stream) == cudaSuccess &&
         cudaMemsetAsync(m->m, 0, pb, m->stream) == cudaSuccess &&
         cudaMemsetAsync(m->v, 0, pb, m->stream) == cudaSuccess;
    std::vector<float> nrm(2 * n_in, 0.0f);
    for (int i = 0; i < n_in; ++i) nrm[n_in + i] = 1.0f;
    ok = ok && cudaMemcpy(m->norm, nrm.data(), nrm.size() * sizeof(float), cudaMemcpyHostToDevice) == cudaSuccess;
    ok = ok && cudaFuncSetAttribute(k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    FwdSmem::BYTES) == cudaSuccess;
    ok = ok && cudaFuncSetAttribute(k_mlp_backward, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)MlpSmem::BYTES) == cudaSuccess;
  }
  if (ok) {
    k_mlp_to_bf16<<<(unsigned)((kW * n_in + kW * kW + kW + 255) / 256), 256, 0, m->stream>>>(m->theta, m->wbf, n_in);
    ok = cudaGetLastError() == cudaSuccess;
  }
  if (!ok) {
    pm_mlp_free(m);
    return PM_ERR_ALLOC;
  }
  *out = m;
  return PM_OK;
}

void pm_mlp_free(pm_mlp* m) {
  if (!m) return;
  void* ptrs[] = {m->theta, m->m, m->v, m->grad, m->partial, m->wbf, m->norm};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  delete m;
}

int64_t pm_mlp_param_count(const pm_mlp* m) { return m ? m->P : 0; }

int pm_mlp_set_params(pm_mlp* m, const float* host_params) {
  if (!m || !host_params) return PM_ERR_INVALID;
  const size_t pb = (size_t)m->P * sizeof(float);
  if (cudaMemcpyAsync(m->theta, host_params, pb, cudaMemcpyHostToDevice, m->stream) != cudaSuccess)
    return PM_ERR_CUDA;
  if (cudaMemsetAsync(m->m, 0, pb, m->stream) != cudaSuccess || cudaMemsetAsync(m->v, 0, pb, m->stream) != cudaSuccess)
    return PM_ERR_CUDA;
  m->step = 0;
  k_mlp_to_bf16<<<(unsigned)((kW * m->n_in + kW * kW + kW + 255) / 256), 256, 0, m->stream>>>(m->theta, m->wbf,
                                                                                              m->n_in);
  if (cudaGetLastError() != cudaSuccess) return PM_ERR_CUDA;
  return mlp_check(cudaStreamSynchronize(m->stream));
}

int pm_mlp_get_params(const pm_mlp* m, float* host_params) {
  if (!m || !host_params) return PM_ERR_INVALID;
  if (cudaMemcpyAsync(host_params, m->theta, (size_t)m->P * sizeof(float), cudaMemcpyDeviceToHost, m->stream) !=
      cudaSuccess)
    return PM_ERR_CUDA;
  return mlp_check(cudaStreamSynchronize(m->stream));
}

int pm_mlp_set_norm(pm_mlp* m, const float* mu, const float* sigma, float y_mu, float y_sigma) {
  if (!m || !mu || !sigma) return PM_ERR_INVALID;
  for (int i = 0; i < m->n_in; ++i)
    if (!(sigma[i] > 0.0f)) return PM_ERR_INVALID;
  if (!(y_sigma > 0.0f)) return PM_ERR_INVALID;
  std::vector<float> nrm(2 * m->n_in);
  memcpy(nrm.data(), mu, m->n_in * sizeof(float));
  memcpy(nrm.data() + m->n_in, sigma, m->n_in * sizeof(float));
  if (cudaMemcpy(m->norm, nrm.data(), nrm.size() * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess)
    return PM_ERR_CUDA;
  m->y_mu = y_mu;
  m->y_sig = y_sigma;
  return PM_OK;
}

int pm_mlp_forward(pm_mlp* m, const float* X, int64_t n, float* y) {
  return m ? mlp_forward_on(m, X, n, y, m->stream) : PM_ERR_INVALID;
}

int pm_mlp_grad(pm_mlp* m, const float* X, const float* y, int64_t n, float* grad, float* loss) {
  if (!m || n <= 0 || !X || !y) return PM_ERR_INVALID;
  return mlp_grad_launch(m, X, y, n, grad, loss);
}

int pm_mlp_train_step(pm_mlp* m, const float* X, const float* y, int64_t n, float lr, float* loss) {
  if (!m || n <= 0 || !X || !y || !(lr > 0.0f)) return PM_ERR_INVALID;
  int rc = mlp_grad_launch(m, X, y, n, m->grad, loss);
  if (rc != PM_OK) return rc;
  m->step += 1;
  const double b1 = 0.9, b2 = 0.999;
  const float bc1 = (float)(1.0 - pow(b1, (double)m->step)), bc2 = (float)(1.0 - pow(b2, (double)m->step));
  k_mlp_adam<<<(unsigned)((m->P + 255) / 256), 256, 0, m->stream>>>(m->theta, m->grad, m->m, m->v, m->P, lr, (float)b1,
                                                                  (float)b2, 1e-8f, bc1, bc2, m->wbf, m->n_in);
  return mlp_check(cudaGetLastError());
}

}  // extern "C"
