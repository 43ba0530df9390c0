// Learned ghost-trace predictor: a small MLP, 4 inputs -> 64 -> 64 -> 1, tanh hidden
// activations, BF16 weights read into FP32 and FP32 accumulation everywhere.  Kernels for
// the mean-squared-error gradient of a sample set (forward + backward) and inference, with the
// hidden layer's products on the tensor cores, and an Adam step on FP32 master weights that
// refreshes their BF16 copy.
//
// Parameter layout (kMlpParams = 4545 values):
//   W1[64][4] | b1[64] | W2[64][64] | b2[64] | w3[64] | b3
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>

#include "../../include/adg.h"
#include "mlp.cuh"

namespace adg {
void noalloc_set_error(const char* msg);

namespace {

// ---- BF16 tensor-core products of FP32 values ------------------------------------------
// The 64 x 64 hidden layer of 16 samples is a [16 x 64] x [64 x 64] product: warp-level BF16
// MMAs (mma.sync m16n8k16, FP32 accumulation).  The BF16 weights enter exactly; FP32 values are
// split into three BF16 terms h = h0 + h1 + h2 (each the BF16 rounding of what the previous
// terms leave; residual below 2^-24 |h|), so a product with the weights keeps FP32 accuracy
// at three MMAs per k-step, and a product of two FP32 matrices at six (the terms of relative
// size down to 2^-16; the rest is below 2^-24).  The 4 -> 64 input layer, the tanh
// activations and the 64 -> 1 output layer stay on the FP32 pipe.
//
// Fragment layouts of mma.m16n8k16 (PTX ISA; g = lane / 4, t = lane % 4):
//   A (16 x 16, row-major, 4 x b32 = 8 bf16): reg 0 = rows g, cols 2t, 2t+1; reg 1 = row g+8;
//     reg 2 = row g, cols 2t+8, 2t+9; reg 3 = row g+8, cols 2t+8, 2t+9 (lower half first)
//   B (16 x 8, column-major, 2 x b32): reg 0 = rows (k) 2t, 2t+1 of column (n) g; reg 1 =
//     rows 2t+8, 2t+9
//   C/D (16 x 8, f32): c0, c1 = row g, cols 2t, 2t+1; c2, c3 = row g+8

// two values rounded to BF16 (nearest even), the first in the lower half
__device__ __forceinline__ unsigned pack_bf16(float lo_col, float hi_col) {
  unsigned r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi_col), "f"(lo_col));
  return r;
}

// three-term BF16 split of two adjacent values into three packed registers
__device__ __forceinline__ void split3(float a, float b, unsigned& r0, unsigned& r1, unsigned& r2) {
  r0 = pack_bf16(a, b);
  const float ar = a - __uint_as_float(r0 << 16);  // exact (Sterbenz)
  const float br = b - __uint_as_float(r0 & 0xFFFF0000u);
  r1 = pack_bf16(ar, br);
  r2 = pack_bf16(ar - __uint_as_float(r1 << 16), br - __uint_as_float(r1 & 0xFFFF0000u));
}

__device__ __forceinline__ void mma_bf16(float (&c)[4], const unsigned (&a)[4], unsigned b0,
                                         unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
      "{%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// c += a b with the product rounded like an FP32 sum: the tensor cores add to their accumulator
// with truncation, so a long sum is kept outside of it.
__device__ __forceinline__ void mma_add(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  float p[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  mma_bf16(p, a, b0, b1);
#pragma unroll
  for (int q = 0; q < 4; ++q) c[q] += p[q];
}
// Sum of products of a three-term FP32 fragment with BF16 weights: leading terms in `c`, the
// others (2^-8 of them and less, where the truncation does not show) in `low`.
__device__ __forceinline__ void mma_split(float (&c)[4], float (&low)[4], const unsigned (&a)[3][4],
                                          unsigned b0, unsigned b1) {
  mma_bf16(low, a[2], b0, b1);
  mma_bf16(low, a[1], b0, b1);
  mma_add(c, a[0], b0, b1);
}

// four 8 x 8 BF16 tiles from shared memory, transposed; lanes 8m..8m+7 hold the row addresses
// of tile m (16 bytes each, 16-byte aligned)
__device__ __forceinline__ void ldmatrix_trans(unsigned (&r)[4], const uint16_t* row) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((unsigned)__cvta_generic_to_shared(row))
               : "memory");
}

// the same without the transposition
__device__ __forceinline__ void ldmatrix(unsigned (&r)[4], const uint16_t* row) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((unsigned)__cvta_generic_to_shared(row))
               : "memory");
}

// First-layer activations tanh(W1 x + b1) of the 16-column block kk for rows g and g+8: h[row]
// [columns c, c+1, c+8, c+9], c = 16 kk + 2t.  w: W1[64][4] | b1[64], 16-byte aligned.
__device__ __forceinline__ void first_layer(const float* w, const float (&x0)[4], const float (&x1)[4],
                                            int kk, int t, float (&h)[2][4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int c = kk * 16 + 2 * t + (q & 1) + (q >> 1) * 8;
    const float4 w1 = *reinterpret_cast<const float4*>(w + kW1 + c * 4);
    const float wc[4] = {w1.x, w1.y, w1.z, w1.w};
    float z0 = w[kB1 + c], z1 = w[kB1 + c];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      z0 = fmaf(wc[i], x0[i], z0);
      z1 = fmaf(wc[i], x1[i], z1);
    }
    h[0][q] = tanhf(z0);
    h[1][q] = tanhf(z1);
  }
}

// A fragments (three terms) of the values v[row][columns c, c+1, c+8, c+9]
__device__ __forceinline__ void split_fragment(const float (&v)[2][4], unsigned (&a)[3][4]) {
  split3(v[0][0], v[0][1], a[0][0], a[1][0], a[2][0]);
  split3(v[1][0], v[1][1], a[0][1], a[1][1], a[2][1]);
  split3(v[0][2], v[0][3], a[0][2], a[1][2], a[2][2]);
  split3(v[1][2], v[1][3], a[0][3], a[1][3], a[2][3]);
}

// ---- gradient ------------------------------------------------------------------------
// A block takes chunks of 128 samples, 16 per warp: forward pass, error and backward pass in
// registers (z2 = h1 W2^T and dh1 = dz2 W2 on the tensor cores), the BF16 terms of h1 and dz2
// and the FP32 dz1 into shared memory; then the block forms dW2 = dz2^T h1 on the tensor cores
// (each warp a 16 x 32 part of it, its sum over the chunks in registers) and dW1, db1 on the
// FP32 pipe.  Bound by latency at 8 warps per SM.  65536 samples with the Adam step: 219 -> 46 us
// against one sample per thread with every product a chain of shared-memory operands; errors
// against 64 bits unchanged.
constexpr int kSamples = 128;   // samples per chunk
constexpr int kGradThreads = 256;
constexpr int kPitch = 72;      // BF16 row pitch: 16-byte rows, 8 rows in distinct banks
constexpr int kZPitch = 65;     // FP32 row pitch of dz1

struct GradSmem {
  uint16_t h1[3][kSamples][kPitch];
  uint16_t d2[3][kSamples][kPitch];
  uint16_t w2[64][kPitch];   // [out][in]
  uint16_t w2t[64][kPitch];  // [in][out]
  float z1[kSamples][kZPitch];
  float x[kSamples][4];
  float w1[kW2];             // W1 | b1
  float wo[kMlpParams - kB2];  // b2 | w3 | b3
};

__global__ void __launch_bounds__(kGradThreads)
mlp_grad_kernel(const uint16_t* __restrict__ pbf, const float* __restrict__ x,
                const float* __restrict__ target, unsigned n, float inv_n, float* __restrict__ grad,
                float* __restrict__ loss) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  GradSmem& S = *reinterpret_cast<GradSmem*>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  for (int i = tid; i < kW2; i += kGradThreads) S.w1[i] = bf16_to_float(pbf[i]);
  for (int i = tid; i < kMlpParams - kB2; i += kGradThreads) S.wo[i] = bf16_to_float(pbf[kB2 + i]);
  for (int i = tid; i < 64 * 64; i += kGradThreads) {
    const uint16_t w = pbf[kW2 + i];
    S.w2[i >> 6][i & 63] = w;
    S.w2t[i & 63][i >> 6] = w;
  }
  // this thread's sums over all chunks: dW2 part; db2 and dw3 of the columns 8j + 2t + q; dW1
  // and db1 of unit tid % 64 over a quarter of each chunk; db3 and the loss
  float gw2[4][4], gb2[8][2], gw3[8][2], gw1[5], gb3 = 0.0f, lacc = 0.0f;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int q = 0; q < 4; ++q) gw2[i][q] = 0.0f;
#pragma unroll
  for (int j = 0; j < 8; ++j)
#pragma unroll
    for (int q = 0; q < 2; ++q) gb2[j][q] = gw3[j][q] = 0.0f;
#pragma unroll
  for (int i = 0; i < 5; ++i) gw1[i] = 0.0f;
  const int m0 = (warp & 3) * 16, i0 = (warp >> 2) * 32;  // dW2 rows (out) and columns (in)
  __syncthreads();

  // (sample numbers are unsigned: the last chunk of 2^31 - 1 samples ends beyond them)
  const int chunks = (int)((n + kSamples - 1) / kSamples);
  for (int c = blockIdx.x; c < chunks; c += gridDim.x) {
    const int row0 = warp * 16 + g, row1 = row0 + 8;  // rows within the chunk
    const unsigned s0 = (unsigned)c * kSamples + row0, s1 = s0 + 8;
    float x0[4], x1[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      x0[i] = s0 < n ? x[(size_t)s0 * 4 + i] : 0.0f;
      x1[i] = s1 < n ? x[(size_t)s1 * 4 + i] : 0.0f;
    }
    if (t == 0) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        S.x[row0][i] = x0[i];
        S.x[row1][i] = x1[i];
      }
    }
    // forward
    float f1[4][2][4];  // 1 - h1^2
    float acc[8][4], low[8][4];
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[j][q] = low[j][q] = 0.0f;
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      float h[2][4];
      first_layer(S.w1, x0, x1, kk, t, h);
      unsigned a[3][4];
      split_fragment(h, a);
      const int col = kk * 16 + 2 * t;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        *reinterpret_cast<unsigned*>(&S.h1[k][row0][col]) = a[k][0];
        *reinterpret_cast<unsigned*>(&S.h1[k][row1][col]) = a[k][1];
        *reinterpret_cast<unsigned*>(&S.h1[k][row0][col + 8]) = a[k][2];
        *reinterpret_cast<unsigned*>(&S.h1[k][row1][col + 8]) = a[k][3];
      }
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) f1[kk][r][q] = fmaf(-h[r][q], h[r][q], 1.0f);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const unsigned b0 = *reinterpret_cast<const unsigned*>(&S.w2[j * 8 + g][col]);
        const unsigned b1 = *reinterpret_cast<const unsigned*>(&S.w2[j * 8 + g][col + 8]);
        mma_split(acc[j], low[j], a, b0, b1);
      }
    }
    float y0 = 0.0f, y1 = 0.0f;
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int u = j * 8 + 2 * t + q;
        const float w3 = S.wo[kW3 - kB2 + u], b2 = S.wo[u];
        acc[j][q] = tanhf((acc[j][q] + low[j][q]) + b2);
        acc[j][2 + q] = tanhf((acc[j][2 + q] + low[j][2 + q]) + b2);
        y0 = fmaf(w3, acc[j][q], y0);
        y1 = fmaf(w3, acc[j][2 + q], y1);
      }
    y0 += __shfl_xor_sync(0xffffffffu, y0, 1);
    y0 += __shfl_xor_sync(0xffffffffu, y0, 2);
    y1 += __shfl_xor_sync(0xffffffffu, y1, 1);
    y1 += __shfl_xor_sync(0xffffffffu, y1, 2);
    // error, output-layer gradients, dz2 (in place of the activations)
    const float b3 = S.wo[kB3 - kB2];
    const float e0 = s0 < n ? y0 + b3 - target[s0] : 0.0f, e1 = s1 < n ? y1 + b3 - target[s1] : 0.0f;
    const float dy0 = 2.0f * e0 * inv_n, dy1 = 2.0f * e1 * inv_n;
    if (t == 0) {
      lacc = fmaf(e0 * e0, inv_n, fmaf(e1 * e1, inv_n, lacc));
      gb3 += dy0 + dy1;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const float w3 = S.wo[kW3 - kB2 + j * 8 + 2 * t + q];
        const float h0 = acc[j][q], h1 = acc[j][2 + q];
        gw3[j][q] = fmaf(dy0, h0, fmaf(dy1, h1, gw3[j][q]));
        acc[j][q] = dy0 * w3 * fmaf(-h0, h0, 1.0f);
        acc[j][2 + q] = dy1 * w3 * fmaf(-h1, h1, 1.0f);
        gb2[j][q] += acc[j][q] + acc[j][2 + q];
      }
    // backward through W2
    float dh[8][4];
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) dh[j][q] = low[j][q] = 0.0f;
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      const float v[2][4] = {{acc[2 * kk][0], acc[2 * kk][1], acc[2 * kk + 1][0], acc[2 * kk + 1][1]},
                             {acc[2 * kk][2], acc[2 * kk][3], acc[2 * kk + 1][2], acc[2 * kk + 1][3]}};
      unsigned a[3][4];
      split_fragment(v, a);
      const int col = kk * 16 + 2 * t;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        *reinterpret_cast<unsigned*>(&S.d2[k][row0][col]) = a[k][0];
        *reinterpret_cast<unsigned*>(&S.d2[k][row1][col]) = a[k][1];
        *reinterpret_cast<unsigned*>(&S.d2[k][row0][col + 8]) = a[k][2];
        *reinterpret_cast<unsigned*>(&S.d2[k][row1][col + 8]) = a[k][3];
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const unsigned b0 = *reinterpret_cast<const unsigned*>(&S.w2t[j * 8 + g][col]);
        const unsigned b1 = *reinterpret_cast<const unsigned*>(&S.w2t[j * 8 + g][col + 8]);
        mma_split(dh[j], low[j], a, b0, b1);
      }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int u = j * 8 + 2 * t + q, f = (j & 1) * 2 + q;
        S.z1[row0][u] = (dh[j][q] + low[j][q]) * f1[j >> 1][0][f];
        S.z1[row1][u] = (dh[j][2 + q] + low[j][2 + q]) * f1[j >> 1][1][f];
      }
    __syncthreads();
    // dW2 += dz2^T h1 over the chunk's samples: the chunk's sum, then into gw2
    float cw2[4][4], lw2[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int q = 0; q < 4; ++q) cw2[i][q] = lw2[i][q] = 0.0f;
#pragma unroll 2
    for (int k0 = 0; k0 < kSamples; k0 += 16) {
      const int r = lane & 7, m = lane >> 3;
      unsigned a[3][4];
#pragma unroll
      for (int k = 0; k < 3; ++k)
        ldmatrix_trans(a[k], &S.d2[k][k0 + (m >> 1) * 8 + r][m0 + (m & 1) * 8]);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        unsigned b[3][4];
#pragma unroll
        for (int k = 0; k < 3; ++k)
          ldmatrix_trans(b[k], &S.h1[k][k0 + (m & 1) * 8 + r][i0 + h * 16 + (m >> 1) * 8]);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          float(&l)[4] = lw2[h * 2 + s];
          mma_bf16(l, a[2], b[0][2 * s], b[0][2 * s + 1]);
          mma_bf16(l, a[0], b[2][2 * s], b[2][2 * s + 1]);
          mma_bf16(l, a[1], b[1][2 * s], b[1][2 * s + 1]);
          mma_bf16(l, a[1], b[0][2 * s], b[0][2 * s + 1]);
          mma_bf16(l, a[0], b[1][2 * s], b[1][2 * s + 1]);
          mma_add(cw2[h * 2 + s], a[0], b[0][2 * s], b[0][2 * s + 1]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int q = 0; q < 4; ++q) gw2[i][q] += cw2[i][q] + lw2[i][q];
    // dW1, db1: unit tid % 64, a quarter of the samples; the chunk's sum in two halves
    {
      const int u = tid & 63, q0 = (tid >> 6) * (kSamples / 4);
      float part[2][5] = {};
#pragma unroll 4
      for (int q = q0; q < q0 + kSamples / 4; q += 2) {
#pragma unroll
        for (int o = 0; o < 2; ++o) {
          const float z = S.z1[q + o][u];
          const float4 xv = *reinterpret_cast<const float4*>(S.x[q + o]);
          part[o][0] = fmaf(z, xv.x, part[o][0]);
          part[o][1] = fmaf(z, xv.y, part[o][1]);
          part[o][2] = fmaf(z, xv.z, part[o][2]);
          part[o][3] = fmaf(z, xv.w, part[o][3]);
          part[o][4] += z;
        }
      }
#pragma unroll
      for (int i = 0; i < 5; ++i) gw1[i] += part[0][i] + part[1][i];
    }
    __syncthreads();
  }

  // sums of the block into the gradient
#pragma unroll
  for (int h = 0; h < 4; ++h)
#pragma unroll
    for (int q = 0; q < 4; ++q)
      atomicAdd(&grad[kW2 + (m0 + g + (q >> 1) * 8) * 64 + i0 + h * 8 + 2 * t + (q & 1)], gw2[h][q]);
  // (one addition per block and parameter: more of them would add their rounding errors)
  float* red = &S.z1[0][0];  // [warp][128 + 2]: db2 | dw3 | db3, loss
  float* red1 = red + kGradThreads / 32 * 130;  // [quarter][dW1 | db1]
  {
    const int u = tid & 63, o = (tid >> 6) * 320;
#pragma unroll
    for (int i = 0; i < 4; ++i) red1[o + u * 4 + i] = gw1[i];
    red1[o + 256 + u] = gw1[4];
  }
  // over the rows g of a warp by shuffles, over the warps by shared memory
#pragma unroll
  for (int j = 0; j < 8; ++j)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      float vb = gb2[j][q], vw = gw3[j][q];
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) {
        vb += __shfl_xor_sync(0xffffffffu, vb, o);
        vw += __shfl_xor_sync(0xffffffffu, vw, o);
      }
      if (g == 0) {
        red[warp * 130 + j * 8 + 2 * t + q] = vb;
        red[warp * 130 + 64 + j * 8 + 2 * t + q] = vw;
      }
    }
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    gb3 += __shfl_xor_sync(0xffffffffu, gb3, o);
    lacc += __shfl_xor_sync(0xffffffffu, lacc, o);
  }
  if (lane == 0) {
    red[warp * 130 + 128] = gb3;
    red[warp * 130 + 129] = lacc;
  }
  __syncthreads();
  for (int i = tid; i < 320; i += kGradThreads)  // W1 | b1
    atomicAdd(&grad[kW1 + i], (red1[i] + red1[320 + i]) + (red1[640 + i] + red1[960 + i]));
  if (tid < 130) {
    float v = 0.0f;
#pragma unroll
    for (int w = 0; w < kGradThreads / 32; ++w) v += red[w * 130 + tid];
    // b2 | w3 | b3 follow one another in the parameters
    atomicAdd(tid < 129 ? &grad[kB2 + tid] : loss, v);
  }
}

// ---- inference -------------------------------------------------------------------------
constexpr int kInferWarps = 4;
constexpr int kInferBlocks = 7;  // per SM (72 registers; at 8 it spills, 9 are 13 % slower)

// A warp per 16 samples.  Bound by the issue of the tanh code; the hidden layer's weights were
// it before: rows of 128 bytes put the eight rows of a B fragment on the same banks (8-fold
// conflicts, 72 % of the time in shared-memory wavefronts).  Padded rows and ldmatrix, two
// column blocks each: 1.97 M samples 456 -> 239 us, 65536 25 -> 15.5 us, the same bits.
__global__ void __launch_bounds__(32 * kInferWarps, kInferBlocks)
mlp_forward_mma_kernel(const uint16_t* __restrict__ pbf, const float* __restrict__ x, unsigned n,
                       float* __restrict__ y) {
  __shared__ __align__(16) float Wf[kW2];               // W1 | b1 (FP32)
  __shared__ __align__(16) float Wo[kMlpParams - kB2];  // b2 | w3 | b3 (FP32)
  __shared__ __align__(16) uint16_t W2[64][kPitch];     // [out][in], BF16
  for (int i = threadIdx.x; i < kW2; i += blockDim.x) Wf[i] = bf16_to_float(pbf[i]);
  for (int i = threadIdx.x; i < kMlpParams - kB2; i += blockDim.x) Wo[i] = bf16_to_float(pbf[kB2 + i]);
  for (int i = threadIdx.x; i < 64 * 64; i += blockDim.x) W2[i >> 6][i & 63] = pbf[kW2 + i];
  __syncthreads();
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  // B fragments of two 8-column blocks per ldmatrix: tile m = lane / 8 holds the rows (outputs)
  // of block m / 2 and the inputs 8 (m % 2) to 8 (m % 2) + 7 of the k-step
  const uint16_t* w2row = &W2[(lane >> 4) * 8 + (lane & 7)][((lane >> 3) & 1) * 8];
  const int tiles = (int)((n + 15) / 16);  // (sample numbers unsigned, as in mlp_grad_kernel)
  for (int tile = blockIdx.x * kInferWarps + (threadIdx.x >> 5); tile < tiles;
       tile += gridDim.x * kInferWarps) {
    const unsigned r0 = (unsigned)tile * 16 + g, r1 = r0 + 8;
    float x0[4], x1[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      x0[i] = r0 < n ? x[(size_t)r0 * 4 + i] : 0.0f;
      x1[i] = r1 < n ? x[(size_t)r1 * 4 + i] : 0.0f;
    }
    float acc[8][4];
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[j][q] = 0.0f;
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      float h[2][4];
      first_layer(Wf, x0, x1, kk, t, h);
      unsigned a[3][4];
      split_fragment(h, a);
#pragma unroll
      for (int j = 0; j < 8; j += 2) {
        unsigned b[4];
        ldmatrix(b, w2row + j * 8 * kPitch + kk * 16);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          mma_bf16(acc[j + i], a[0], b[2 * i], b[2 * i + 1]);
          mma_bf16(acc[j + i], a[1], b[2 * i], b[2 * i + 1]);
          mma_bf16(acc[j + i], a[2], b[2 * i], b[2 * i + 1]);
        }
      }
    }
    // second activation and the output layer: this lane holds columns 2t, 2t+1 of each
    // 8-column block for rows r0 (acc[j][0..1]) and r1 (acc[j][2..3])
    float y0 = 0.0f, y1 = 0.0f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int c = j * 8 + 2 * t;
      const float2 b2 = *reinterpret_cast<const float2*>(&Wo[c]);
      const float2 w3 = *reinterpret_cast<const float2*>(&Wo[kW3 - kB2 + c]);
      y0 = fmaf(w3.x, tanhf(acc[j][0] + b2.x), y0);
      y1 = fmaf(w3.x, tanhf(acc[j][2] + b2.x), y1);
      y0 = fmaf(w3.y, tanhf(acc[j][1] + b2.y), y0);
      y1 = fmaf(w3.y, tanhf(acc[j][3] + b2.y), y1);
    }
    y0 += __shfl_xor_sync(0xffffffffu, y0, 1);
    y0 += __shfl_xor_sync(0xffffffffu, y0, 2);
    y1 += __shfl_xor_sync(0xffffffffu, y1, 1);
    y1 += __shfl_xor_sync(0xffffffffu, y1, 2);
    if (t == 0) {
      const float b3 = Wo[kB3 - kB2];
      if (r0 < n) y[r0] = y0 + b3;
      if (r1 < n) y[r1] = y1 + b3;
    }
  }
}

// Adam (Kingma & Ba 2015) on the FP32 master weights; refreshes the BF16 copy and clears
// the gradient for the next accumulation.
__global__ void mlp_adam_kernel(float* __restrict__ p, uint16_t* __restrict__ pbf,
                                float* __restrict__ g, float* __restrict__ m,
                                float* __restrict__ v, float lr, float b1, float b2, float eps,
                                float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= kMlpParams) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.0f - b1) * gi;
  const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  p[i] = pi;
  pbf[i] = float_to_bf16(pi);
  g[i] = 0.0f;
}

__global__ void to_bf16_kernel(const float* __restrict__ p, uint16_t* __restrict__ pbf, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) pbf[i] = float_to_bf16(p[i]);
}

}  // namespace

cudaError_t mlp_infer(const uint16_t* params, const float* x, int64_t n, float* y, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int64_t tiles = (n + 15) / 16;
  const int64_t want = (tiles + kInferWarps - 1) / kInferWarps;
  const int blocks = (int)(want < 152 * kInferBlocks ? want : 152 * kInferBlocks);
  mlp_forward_mma_kernel<<<blocks, 32 * kInferWarps, 0, s>>>(params, x, (unsigned)n, y);
  return cudaGetLastError();
}

namespace {

adg_status mfail(adg_status st, const std::string& m) {
  noalloc_set_error(m.c_str());
  return st;
}

}  // namespace
}  // namespace adg

using namespace adg;

extern "C" {

adg_status adg_mlp_grad(const uint16_t* params_bf16, const float* x, const float* target,
                        int64_t n, float* grad, float* loss, void* cuda_stream) {
  if (!params_bf16 || !x || !target || !grad || !loss || n < 0)
    return mfail(ADG_ERR_INVALID, "bad arguments");
  if (n == 0) return ADG_OK;
  if (n >= ((int64_t)1 << 31)) return mfail(ADG_ERR_INVALID, "too many samples");
  cudaStream_t s = (cudaStream_t)cuda_stream;
  const size_t smem = sizeof(GradSmem);
  cudaError_t e = cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return mfail(ADG_ERR_CUDA, cudaGetErrorString(e));
  const int chunks = (int)((n + kSamples - 1) / kSamples);
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // blocks of equal numbers of chunks: as few as need the same number of rounds (every block
  // adds its sums to the gradient once, with its rounding)
  const int rounds = (chunks + sms - 1) / sms, grid = (chunks + rounds - 1) / rounds;
  mlp_grad_kernel<<<grid, kGradThreads, smem, s>>>(params_bf16, x, target, (unsigned)n, 1.0f / (float)n, grad, loss);
  e = cudaGetLastError();
  return e == cudaSuccess ? ADG_OK : mfail(ADG_ERR_CUDA, cudaGetErrorString(e));
}

adg_status adg_mlp_forward(const uint16_t* params_bf16, const float* x, int64_t n, float* y,
                           void* cuda_stream) {
  if (!params_bf16 || !x || !y || n < 0) return mfail(ADG_ERR_INVALID, "bad arguments");
  if (n == 0) return ADG_OK;
  if (n >= ((int64_t)1 << 31)) return mfail(ADG_ERR_INVALID, "too many samples");
  cudaError_t e = mlp_infer(params_bf16, x, n, y, (cudaStream_t)cuda_stream);
  return e == cudaSuccess ? ADG_OK : mfail(ADG_ERR_CUDA, cudaGetErrorString(e));
}

adg_status adg_mlp_adam(float* params, uint16_t* params_bf16, float* grad, float* m, float* v,
                        float lr, float beta1, float beta2, float eps, int t, void* cuda_stream) {
  if (!params || !params_bf16 || !grad || !m || !v || t < 1) return mfail(ADG_ERR_INVALID, "bad arguments");
  const float c1 = 1.0f - powf(beta1, (float)t), c2 = 1.0f - powf(beta2, (float)t);
  mlp_adam_kernel<<<(kMlpParams + 255) / 256, 256, 0, (cudaStream_t)cuda_stream>>>(
      params, params_bf16, grad, m, v, lr, beta1, beta2, eps, c1, c2);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? ADG_OK : mfail(ADG_ERR_CUDA, cudaGetErrorString(e));
}

adg_status adg_mlp_to_bf16(const float* params, uint16_t* params_bf16, void* cuda_stream) {
  if (!params || !params_bf16) return mfail(ADG_ERR_INVALID, "bad arguments");
  to_bf16_kernel<<<(kMlpParams + 255) / 256, 256, 0, (cudaStream_t)cuda_stream>>>(params, params_bf16, kMlpParams);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? ADG_OK : mfail(ADG_ERR_CUDA, cudaGetErrorString(e));
}

int adg_mlp_num_params(void) { return kMlpParams; }

}  // extern "C"
