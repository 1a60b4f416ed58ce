// mlp.cu -- the surrogate network of the learned proposal on tensor cores.
//
// s(x) = w3 . tanh(W2^T tanh(W1^T x + b1) + b2) + b3, hidden width 64, with
// bfloat16 operands and FP32 accumulation (mma.sync m16n8k16).  A warp owns
// 16 rows; the accumulator fragments of one layer are re-packed in registers
// as the operand fragments of the next.  Training computes per-CTA partial
// gradients of the mean squared error (the weight gradients are second products
// over the CTA's rows, staged in shared memory) and sums them in a fixed order
// for an Adam step.
// The proposal uses the gradient with respect to the input.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <utility>

#include "common.cuh"
#include "internal.h"

namespace smc2 {

using bf16 = __nv_bfloat16;

constexpr int kRowsCta = 16 * kMlpWarps;  // rows per CTA
constexpr int kLd = kMlpH + 8;             // padded row of 64-wide bf16 tiles (conflict-free fragments)

__host__ __device__ inline int mlp_nparams(int D) { return D * kMlpH + kMlpH * kMlpH + 3 * kMlpH + 1; }
__host__ __device__ inline int off_b1(int D) { return D * kMlpH; }
__host__ __device__ inline int off_W2(int D) { return D * kMlpH + kMlpH; }
__host__ __device__ inline int off_b2(int D) { return off_W2(D) + kMlpH * kMlpH; }
__host__ __device__ inline int off_w3(int D) { return off_b2(D) + kMlpH; }
__host__ __device__ inline int off_b3(int D) { return off_w3(D) + kMlpH; }

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ float round_bf16(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

__device__ __forceinline__ float bf16_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }

// tanh x = sign(x) (1 - e) / (1 + e) with e = exp(-2|x|) in (0, 1]: the
// hardware exp2 (relative error about 2^-22) and reciprocal.  The absolute error
// stays near 2^-22, far below the half step (2^-9 relative) of the bfloat16 the
// activations are rounded to.  A subnormal e or x changes neither 1 - e nor 1 + e.
__device__ __forceinline__ float tanh_act(float x) {
  const float e = ex2_approx(fabsf(x) * -2.8853900817779268f);
  return copysignf((1.f - e) * rcp_approx(1.f + e), x);
}
__device__ __forceinline__ uint32_t ld32(const bf16* p) { return *reinterpret_cast<const uint32_t*>(p); }

// D = A B + D for a 16x16 (row) by 16x8 (column) bf16 product, FP32 accumulators.
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                         uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Four 8x8 bf16 matrices between registers and shared memory (lane l gives the
// address of row l % 8 of matrix l / 8): lane (g, t) holds elements (g, 2t) and
// (g, 2t + 1) of each, or of its transpose.
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const bf16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_addr(p))
               : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const bf16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_addr(p))
               : "memory");
}
__device__ __forceinline__ void ldsm2t(uint32_t& r0, uint32_t& r1, const bf16* p) {  // two: lanes 0-15 address
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n"
               : "=r"(r0), "=r"(r1)
               : "r"(smem_addr(p))
               : "memory");
}
__device__ __forceinline__ void stsm4(bf16* p, const uint32_t (&r)[4]) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1,%2,%3,%4};\n" ::"r"(smem_addr(p)), "r"(r[0]),
               "r"(r[1]), "r"(r[2]), "r"(r[3])
               : "memory");
}
// The two orders in which an operand's four matrices cover a 16x16 tile: the lane's (row, column)
// with matrices 1 and 2 below and right of the first (rows first), or right and below (columns first).
struct LaneTile {
  int lo, hi;  // l % 8 + 8 (l / 8 % 2) and 8 (l / 16); l % 8 + 8 (l / 16) and 8 (l / 8 % 2)
  int lo2, hi2;
  __device__ LaneTile() {
    const int l = threadIdx.x & 31;
    lo = l & 15;
    hi = (l >> 4) * 8;
    lo2 = (l & 7) + (l >> 4) * 8;
    hi2 = ((l >> 3) & 1) * 8;
  }
};

// Shared-memory copy of the operands, padded rows (144 bytes: eight rows of a
// matrix fall in different banks).  Both orientations of a weight matrix come from
// one copy, read with or without a transpose:
//   w1b [16][kLd]   W1 input-major (rows from D on zero)
//   w2b [64][kLd]   W2 input-major
//   w3b [64], b1, b2, w3 in FP32
struct MlpSmemWeights {
  alignas(16) bf16 w1b[16 * kLd];
  alignas(16) bf16 w2b[kMlpH * kLd];
  alignas(16) bf16 w3b[kMlpH];
  alignas(16) float b1[kMlpH];
  float b2[kMlpH], w3f[kMlpH];  // w3f: the bfloat16 w3 as FP32
  float b3;
};

// Load the weights from the FP32 parameter vector (bf16-rounded copies).
// Every thread issues its float4 loads before the first shared-memory store
// (the vector is 16-byte aligned and every block of it starts at a multiple
// of four floats), so a CTA waits for about one L2 round trip.
__device__ void load_weights(MlpSmemWeights& W, const float* p, int D) {
  constexpr int kV = 8;  // float4 loads in flight per thread and round
  const int nt = blockDim.x, tid = threadIdx.x;
  for (int e = D * kLd + tid; e < 16 * kLd; e += nt) W.w1b[e] = __float2bfloat16_rn(0.f);
  const int n4 = (mlp_nparams(D) - 1) / 4;  // float4 blocks before b3
  const float4* p4 = reinterpret_cast<const float4*>(p);
  for (int base = tid; base < n4; base += kV * nt) {
    float4 v[kV];
#pragma unroll
    for (int u = 0; u < kV; ++u) {
      const int q4 = base + u * nt;
      v[u] = q4 < n4 ? p4[q4] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < kV; ++u) {
      const int q4 = base + u * nt;
      if (q4 >= n4) break;
      const float vals[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int q = 4 * q4 + c;
        const float f = vals[c];
        if (q < off_b1(D)) {  // W1[d][o]
          W.w1b[q / kMlpH * kLd + q % kMlpH] = __float2bfloat16_rn(f);
        } else if (q < off_W2(D)) {
          W.b1[q - off_b1(D)] = f;
        } else if (q < off_b2(D)) {  // W2[i][o]
          const int r = q - off_W2(D);
          W.w2b[r / kMlpH * kLd + r % kMlpH] = __float2bfloat16_rn(f);
        } else if (q < off_w3(D)) {
          W.b2[q - off_b2(D)] = f;
        } else {
          const bf16 h = __float2bfloat16_rn(f);  // weights are used rounded, biases exact
          W.w3b[q - off_w3(D)] = h;
          W.w3f[q - off_w3(D)] = __bfloat162float(h);
        }
      }
    }
  }
  if (tid == 0) W.b3 = p[off_b3(D)];
}

// Forward pass of one warp's 16 rows.  Lane (g, t) = (lane / 4, lane % 4)
// holds columns 8j + 2t + {0,1} of rows g and g+8 of every 16x8 tile j; a packed
// operand [kk] holds tiles 2kk and 2kk + 1, rows g and g+8 of each.
struct WarpForward {
  float h1[8][4], h2[8][4];  // tanh activations (FP32)
  uint32_t h1p[4][4];        // h1 packed
  float s_lo, s_hi;          // s of rows g and g+8 (every lane of the quad)
};

__device__ __forceinline__ void pack_tiles(uint32_t (&p)[4], const float (&a)[4], const float (&b)[4]) {
  p[0] = pack_bf16(a[0], a[1]);
  p[1] = pack_bf16(a[2], a[3]);
  p[2] = pack_bf16(b[0], b[1]);
  p[3] = pack_bf16(b[2], b[3]);
}

// xp: the rows' inputs as a packed operand (16 columns, zero weights beyond D)
__device__ __forceinline__ void warp_forward(const MlpSmemWeights& W, const uint32_t (&xp)[4], WarpForward& F) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const LaneTile lt;
  const bf16* w1 = W.w1b + lt.lo * kLd + lt.hi;
  const bf16* w2 = W.w2b + lt.lo * kLd + lt.hi;
#pragma unroll
  for (int jj = 0; jj < 4; ++jj) {
    uint32_t w[4];
    ldsm4t(w, w1 + 16 * jj);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int j = 2 * jj + h;
      float c[4] = {0.f, 0.f, 0.f, 0.f};
      mma_bf16(c, xp[0], xp[1], xp[2], xp[3], w[2 * h], w[2 * h + 1]);
      const float2 b = *reinterpret_cast<const float2*>(W.b1 + 8 * j + 2 * t);
      F.h1[j][0] = tanh_act(c[0] + b.x);
      F.h1[j][1] = tanh_act(c[1] + b.y);
      F.h1[j][2] = tanh_act(c[2] + b.x);
      F.h1[j][3] = tanh_act(c[3] + b.y);
    }
    pack_tiles(F.h1p[jj], F.h1[2 * jj], F.h1[2 * jj + 1]);
  }
  float c3[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int jj = 0; jj < 4; ++jj) {
    float c[2][4];
#pragma unroll
    for (int e = 0; e < 4; ++e) c[0][e] = c[1][e] = 0.f;
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      uint32_t w[4];
      ldsm4t(w, w2 + 16 * kk * kLd + 16 * jj);
      mma_bf16(c[0], F.h1p[kk][0], F.h1p[kk][1], F.h1p[kk][2], F.h1p[kk][3], w[0], w[1]);
      mma_bf16(c[1], F.h1p[kk][0], F.h1p[kk][1], F.h1p[kk][2], F.h1p[kk][3], w[2], w[3]);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int j = 2 * jj + h;
      const float2 b = *reinterpret_cast<const float2*>(W.b2 + 8 * j + 2 * t);
      F.h2[j][0] = tanh_act(c[h][0] + b.x);
      F.h2[j][1] = tanh_act(c[h][1] + b.y);
      F.h2[j][2] = tanh_act(c[h][2] + b.x);
      F.h2[j][3] = tanh_act(c[h][3] + b.y);
    }
    uint32_t hp[4];
    pack_tiles(hp, F.h2[2 * jj], F.h2[2 * jj + 1]);
    const uint32_t b0 = g == 0 ? ld32(W.w3b + 16 * jj + 2 * t) : 0u;
    const uint32_t b1 = g == 0 ? ld32(W.w3b + 16 * jj + 8 + 2 * t) : 0u;
    mma_bf16(c3, hp[0], hp[1], hp[2], hp[3], b0, b1);
  }
  // column 0 of the output tile sits in the lanes with t = 0
  F.s_lo = __shfl_sync(0xffffffffu, c3[0], lane & ~3) + W.b3;
  F.s_hi = __shfl_sync(0xffffffffu, c3[2], lane & ~3) + W.b3;
}

// Back-propagation of the row signals (ga, gb) to dz2 and dz1, both as packed operands.
__device__ __forceinline__ void warp_backward(const MlpSmemWeights& W, const WarpForward& F, float ga,
                                              float gb, uint32_t (&dz2)[4][4], uint32_t (&dz1)[4][4]) {
  const int lane = threadIdx.x & 31, t = lane & 3;
  const LaneTile lt;
  const bf16* w2 = W.w2b + lt.lo2 * kLd + lt.hi2;
#pragma unroll
  for (int jj = 0; jj < 4; ++jj) {
    float z[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int j = 2 * jj + h;
      const float2 w = *reinterpret_cast<const float2*>(W.w3f + 8 * j + 2 * t);
      z[h][0] = ga * w.x * (1.f - F.h2[j][0] * F.h2[j][0]);
      z[h][1] = ga * w.y * (1.f - F.h2[j][1] * F.h2[j][1]);
      z[h][2] = gb * w.x * (1.f - F.h2[j][2] * F.h2[j][2]);
      z[h][3] = gb * w.y * (1.f - F.h2[j][3] * F.h2[j][3]);
    }
    pack_tiles(dz2[jj], z[0], z[1]);
  }
#pragma unroll
  for (int jj = 0; jj < 4; ++jj) {  // dh1 = dz2 W2^T, tiles over the input units
    float c[2][4];
#pragma unroll
    for (int e = 0; e < 4; ++e) c[0][e] = c[1][e] = 0.f;
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      uint32_t w[4];
      ldsm4(w, w2 + 16 * jj * kLd + 16 * kk);
      mma_bf16(c[0], dz2[kk][0], dz2[kk][1], dz2[kk][2], dz2[kk][3], w[0], w[1]);
      mma_bf16(c[1], dz2[kk][0], dz2[kk][1], dz2[kk][2], dz2[kk][3], w[2], w[3]);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float h1 = F.h1[2 * jj + h][e];
        c[h][e] *= 1.f - h1 * h1;
      }
    pack_tiles(dz1[jj], c[0], c[1]);
  }
}
// Element (column 8j + 2t + e % 2, row g + 8 (e / 2)) of a packed operand.
__device__ __forceinline__ float unpack_tile(const uint32_t (&p)[4][4], int j, int e) {
  const uint32_t v = p[j >> 1][2 * (j & 1) + (e >> 1)];
  return (e & 1) ? bf16_hi(v) : bf16_lo(v);
}

// Sum over the eight row groups g of a warp (lanes with equal t).
__device__ __forceinline__ float sum_over_g(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 4);
  v += __shfl_xor_sync(0xffffffffu, v, 8);
  v += __shfl_xor_sync(0xffffffffu, v, 16);
  return v;
}

constexpr int kGradWarps = 8;                            // warps of a training-step CTA
constexpr int kGradTiles = 1;                            // 16-row tiles per warp
constexpr int kRowsGrad = 16 * kGradWarps * kGradTiles;  // rows per CTA
constexpr int kLdR = kRowsGrad + 8;                      // padded row of the staged [unit][row] tiles

struct MlpGradSmem {
  MlpSmemWeights W;
  bf16 h1T[kMlpH * kLdR];                   // [i][row] h1 of the CTA's rows (bf16)
  bf16 dz2T[kMlpH * kLdR];                  // [o][row] dz2 of the CTA's rows (bf16)
  float col[kGradWarps][3][kMlpH];          // per warp: db1, db2, dw3
  float w1g[kGradWarps][kMlpMaxD][kMlpH];   // per warp: dW1
  float sc[kGradWarps][2];                  // per warp: sum e^2, db3
};

// Partial gradients of L = (1/R) sum (s(x_r) - y_r)^2: CTA c writes the
// gradient over its rows (and their sum of e^2) to part[c][0..P].
__global__ void __launch_bounds__(32 * kGradWarps)
    mlp_grad_kernel(const float* __restrict__ p, int D, const float* __restrict__ x,
                    const float* __restrict__ y, int R_imm, const int* R_dev, float* __restrict__ part,
                    int* step) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int R = R_dev ? *R_dev : R_imm;
  const int n_active = (R + kRowsGrad - 1) / kRowsGrad;
  const int P = mlp_nparams(D);
  MlpGradSmem& S = *reinterpret_cast<MlpGradSmem*>(smem_raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  if (step && blockIdx.x == 0 && threadIdx.x == 0) *step += 1;  // the Adam step this gradient feeds
  if ((int)blockIdx.x < n_active) {
    load_weights(S.W, p, D);
    for (int e = threadIdx.x; e < kGradWarps * 3 * kMlpH; e += blockDim.x) (&S.col[0][0][0])[e] = 0.f;
    for (int e = threadIdx.x; e < kGradWarps * kMlpMaxD * kMlpH; e += blockDim.x) (&S.w1g[0][0][0])[e] = 0.f;
    __syncthreads();
    float l_acc = 0.f, d3_acc = 0.f;
    for (int tile = 0; tile < kGradTiles; ++tile) {
      const int rl = (warp * kGradTiles + tile) * 16 + g;  // row within the CTA
      const int ra = blockIdx.x * kRowsGrad + rl, rb = ra + 8;
      const bool va = ra < R, vb = rb < R;
      float xa[4], xb[4], xfa[kMlpMaxD], xfb[kMlpMaxD];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int k = 2 * t + (e & 1) + (e >> 1) * 8;
        xa[e] = (va && k < D) ? x[(size_t)ra * D + k] : 0.f;
        xb[e] = (vb && k < D) ? x[(size_t)rb * D + k] : 0.f;
      }
#pragma unroll
      for (int d = 0; d < kMlpMaxD; ++d) {
        xfa[d] = (va && d < D) ? round_bf16(x[(size_t)ra * D + d]) : 0.f;
        xfb[d] = (vb && d < D) ? round_bf16(x[(size_t)rb * D + d]) : 0.f;
      }
      WarpForward F;
      const uint32_t xp[4] = {pack_bf16(xa[0], xa[1]), pack_bf16(xb[0], xb[1]), pack_bf16(xa[2], xa[3]),
                              pack_bf16(xb[2], xb[3])};
      warp_forward(S.W, xp, F);
      const float ea = va ? F.s_lo - y[ra] : 0.f, eb = vb ? F.s_hi - y[rb] : 0.f;
      const float ga = 2.f * ea / (float)R, gb = 2.f * eb / (float)R;
      uint32_t dz2p[4][4], dz1p[4][4];
      warp_backward(S.W, F, ga, gb, dz2p, dz1p);
      float dz2[8][4], dz1[8][4];
#pragma unroll
      for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          dz2[j][e] = unpack_tile(dz2p, j, e);
          dz1[j][e] = unpack_tile(dz1p, j, e);
        }
      // loss and db3: rows counted once, in the t = 0 lanes
      l_acc += warp_sum(t == 0 ? ea * ea + eb * eb : 0.f);
      d3_acc += warp_sum(t == 0 ? ga + gb : 0.f);
      // column sums over the tile's rows: db2, dw3, db1, dW1 (the warp owns its slots)
#pragma unroll
      for (int j = 0; j < 8; ++j) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int c = 8 * j + 2 * t + e;
          const float v_db2 = sum_over_g(dz2[j][e] + dz2[j][2 + e]);
          const float v_dw3 = sum_over_g(round_bf16(F.h2[j][e]) * ga + round_bf16(F.h2[j][2 + e]) * gb);
          const float v_db1 = sum_over_g(dz1[j][e] + dz1[j][2 + e]);
          if (g == 0) {
            S.col[warp][1][c] += v_db2;
            S.col[warp][2][c] += v_dw3;
            S.col[warp][0][c] += v_db1;
          }
#pragma unroll
          for (int d = 0; d < kMlpMaxD; ++d) {
            if (d >= D) break;
            const float w = sum_over_g(xfa[d] * dz1[j][e] + xfb[d] * dz1[j][2 + e]);
            if (g == 0) S.w1g[warp][d][c] += w;
          }
        }
      }
      // stage h1 and dz2 transposed for dW2 = h1^T dz2 over the CTA's rows
#pragma unroll
      for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int c = 8 * j + 2 * t + e;
          S.h1T[c * kLdR + rl] = __float2bfloat16_rn(F.h1[j][e]);
          S.h1T[c * kLdR + rl + 8] = __float2bfloat16_rn(F.h1[j][2 + e]);
          S.dz2T[c * kLdR + rl] = __float2bfloat16_rn(dz2[j][e]);
          S.dz2T[c * kLdR + rl + 8] = __float2bfloat16_rn(dz2[j][2 + e]);
        }
    }
    if (lane == 0) {
      S.sc[warp][0] = l_acc;
      S.sc[warp][1] = d3_acc;
    }
    __syncthreads();
    float* out = part + (size_t)blockIdx.x * (P + 1);
    {  // dW2: warp (mt, nh) computes units i of m-tile mt against o of n-tiles 4 nh .. 4 nh + 3
      const int mt = warp & 3, nh = warp >> 2;
      float acc[4][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
#pragma unroll 4
      for (int kk = 0; kk < kRowsGrad / 16; ++kk) {
        const bf16* a = S.h1T + (16 * mt + g) * kLdR + 16 * kk + 2 * t;
        const uint32_t a0 = ld32(a), a1 = ld32(a + 8 * kLdR), a2 = ld32(a + 8), a3 = ld32(a + 8 * kLdR + 8);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const bf16* b = S.dz2T + (8 * (4 * nh + j) + g) * kLdR + 16 * kk + 2 * t;
          mma_bf16(acc[j], a0, a1, a2, a3, ld32(b), ld32(b + 8));
        }
      }
      float* gW2 = out + off_W2(D);
      const int i0 = 16 * mt + g;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int o = 8 * (4 * nh + j) + 2 * t;
        gW2[i0 * kMlpH + o] = acc[j][0];
        gW2[i0 * kMlpH + o + 1] = acc[j][1];
        gW2[(i0 + 8) * kMlpH + o] = acc[j][2];
        gW2[(i0 + 8) * kMlpH + o + 1] = acc[j][3];
      }
    }
    // the remaining partials: warp sums in warp order
    for (int e = threadIdx.x; e < kMlpH; e += blockDim.x) {
      float b1s = 0.f, b2s = 0.f, w3s = 0.f;
      for (int w = 0; w < kGradWarps; ++w) {
        b1s += S.col[w][0][e];
        b2s += S.col[w][1][e];
        w3s += S.col[w][2][e];
      }
      out[off_b1(D) + e] = b1s;
      out[off_b2(D) + e] = b2s;
      out[off_w3(D) + e] = w3s;
      for (int d = 0; d < D; ++d) {
        float s1 = 0.f;
        for (int w = 0; w < kGradWarps; ++w) s1 += S.w1g[w][d][e];
        out[d * kMlpH + e] = s1;
      }
    }
    if (threadIdx.x == 0) {
      float l2 = 0.f, b3s = 0.f;
      for (int w = 0; w < kGradWarps; ++w) {
        l2 += S.sc[w][0];
        b3s += S.sc[w][1];
      }
      out[off_b3(D)] = b3s;
      out[P] = l2;
    }
  }
}

// Sum of the partials over the CTAs in order, then the loss (and the gradient
// when grad != nullptr) and, with adam != 0, one Adam step on p (moments m, v;
// *step, already advanced by the gradient kernel, is the step number).
__global__ void __launch_bounds__(128)
    mlp_reduce_kernel(float* p, int D, const float* __restrict__ part, int R_imm, const int* R_dev,
                      float* grad, float* loss, int adam, float* m, float* v, int* step, float lr) {
  const int P = mlp_nparams(D);
  const int R = R_dev ? *R_dev : R_imm;
  const int n = (R + kRowsGrad - 1) / kRowsGrad;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q > P) return;
  float sum = 0.f;
  for (int c0 = 0; c0 < n; c0 += 16) {
    float tv[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) tv[u] = c0 + u < n ? __ldcg(part + (size_t)(c0 + u) * (P + 1) + q) : 0.f;
#pragma unroll
    for (int u = 0; u < 16; ++u) sum += tv[u];
  }
  if (q == P) {
    if (loss) loss[0] = R > 0 ? sum / (float)R : 0.f;
    return;
  }
  if (grad) grad[q] = sum;
  if (!adam) return;
  const float beta1 = 0.9f, beta2 = 0.999f, eps = 1e-8f;
  const float mq = beta1 * m[q] + (1.f - beta1) * sum;
  const float vq = beta2 * v[q] + (1.f - beta2) * sum * sum;
  m[q] = mq;
  v[q] = vq;
  const float t_step = (float)*step;
  const float bc1 = 1.f - powf(beta1, t_step), bc2 = 1.f - powf(beta2, t_step);
  p[q] -= lr * (mq / bc1) / (sqrtf(vq / bc2) + eps);
}

// ---------------------------------------------------------------------------
// training: all Adam steps of one call in one launch of a thread-block cluster
// ---------------------------------------------------------------------------
// The cluster's CTAs split the rows; each keeps the bfloat16 weights, the FP32
// biases, its rows and its partial gradient in shared memory, so the kernel
// body, the weights and the data stay on the SMs for every step.  Per step:
// partial gradients over the CTA's rows; cluster barrier; CTA c sums parameter
// slice c over the cluster's CTAs in rank order (distributed shared memory),
// takes the Adam step on it -- the FP32 parameters and moments of a thread's
// pair stay in its registers -- and writes the new operands into every CTA's
// copy; cluster barrier.
// A step is bound by latency and by the two hardware approximations of each
// tanh (65,536 of 256 rows and 128 units, at 16 a clock and SM: 2.1 us), so
// sixteen warps take one 16-row tile each and every operand moves as four 8x8
// matrices an instruction (eight warps with two tiles each in turn, operands and
// staged transposes by 4- and 2-byte accesses: 13.5 us a step, this form 9.7; the
// standardisation, with one thread a total reading the other CTAs, 34 -> 14.5 us a
// call).  4096 rows, D = 4, 16 steps: 253 -> 172 us.
constexpr int kTrainWarps = 16;
constexpr int kMaxCluster = 16;               // CTAs of the training cluster, at most
constexpr int kTrainRows = 16 * kTrainWarps;  // rows per chunk: one 16-row tile per warp
constexpr int kLdT = kTrainRows + 8;          // padded row of the inputs' [coordinate][row] tile
constexpr int kMlpPmax = kMlpMaxD * kMlpH + kMlpH * kMlpH + 3 * kMlpH + 1;
constexpr int kStdWarps = 8;                  // warps that sum in the standardisation

struct MlpTrainSmem {
  MlpSmemWeights W;
  alignas(16) bf16 h1[kTrainRows * kLd];      // [row][unit] h1 of the chunk's rows
  alignas(16) bf16 dz2[kTrainRows * kLd];     // [row][unit] dz2
  alignas(16) bf16 dz1[kTrainRows * kLd];     // [row][unit] dz1
  alignas(16) bf16 xT[16 * kLdT];             // [d][row] inputs (bf16), row D all ones, rest zero
  alignas(16) float gp[kMlpPmax + 1];         // partial gradient over the CTA's rows, then sum e^2
  float ys[kTrainRows];                       // the chunk's targets
  float col[kTrainWarps][kMlpH];              // per warp: dw3 of its tile
  float pairs[kTrainWarps / 2][kMlpH];        // per two warps: dw3 over the chunks
  float sc[kTrainWarps][2];                   // per warp: sum e^2, db3 of its tile
  float psc[kTrainWarps / 2][2];              // per two warps, over the chunks
  float wred[kStdWarps][2 * kMlpMaxD + 1];    // block reductions: per-warp values
  float cred[2][2 * kMlpMaxD + 1];            // the CTA's totals, read by the cluster (in turn)
  float tot[2 * kMlpMaxD + 1];                // the cluster's totals
};

// Totals over the cluster of NV values per thread of the first kStdWarps warps (sums, or
// maxima), in a fixed order: warp shuffles, the warps in order, then the CTAs in rank order
// through distributed shared memory.  Every thread of every CTA gets them.  Calls use cred
// in turn (n counts them): a CTA writes a buffer again only after a later call's barrier,
// which every reader of the earlier call has passed.
template <int NV>
__device__ void cluster_totals(float (&v)[NV], MlpTrainSmem& S, cooperative_groups::cluster_group& cluster,
                               bool is_max, int& n) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = threadIdx.x;
  float* cred = S.cred[n & 1];
  ++n;
  if (warp < kStdWarps) {
#pragma unroll
    for (int u = 0; u < NV; ++u) {
      const float r = is_max ? warp_max(v[u]) : warp_sum(v[u]);
      if (lane == 0) S.wred[warp][u] = r;
    }
  }
  __syncthreads();
  if (i < NV) {
    float r = S.wred[0][i];
    for (int w = 1; w < kStdWarps; ++w) r = is_max ? fmaxf(r, S.wred[w][i]) : r + S.wred[w][i];
    cred[i] = r;
  }
  cluster.sync();
  const int C = (int)cluster.num_blocks();
  if (i < NV) {
    float u[kMaxCluster];
#pragma unroll
    for (int q = 0; q < kMaxCluster; ++q) u[q] = q < C ? cluster.map_shared_rank(cred, q)[i] : 0.f;
    float r = u[0];
#pragma unroll
    for (int q = 1; q < kMaxCluster; ++q)
      if (q < C) r = is_max ? fmaxf(r, u[q]) : r + u[q];
    S.tot[i] = r;
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < NV; ++u) v[u] = S.tot[u];
}

// The operand copies of parameters q and q + 1 (q even; the blocks are even, so both are of one
// block) into one CTA's shared memory.  q = P - 1 (b3) has no second.
__device__ __forceinline__ void put_weights(MlpSmemWeights& W, int D, int q, float2 p) {
  if (q >= off_W2(D) && q < off_b2(D)) {
    const int r = q - off_W2(D);
    *reinterpret_cast<uint32_t*>(W.w2b + r / kMlpH * kLd + r % kMlpH) = pack_bf16(p.x, p.y);
  } else if (q < off_b1(D)) {
    *reinterpret_cast<uint32_t*>(W.w1b + q / kMlpH * kLd + q % kMlpH) = pack_bf16(p.x, p.y);
  } else if (q < off_W2(D)) {
    *reinterpret_cast<float2*>(W.b1 + (q - off_b1(D))) = p;
  } else if (q < off_w3(D)) {
    *reinterpret_cast<float2*>(W.b2 + (q - off_b2(D))) = p;
  } else if (q < off_b3(D)) {
    const uint32_t h = pack_bf16(p.x, p.y);
    *reinterpret_cast<uint32_t*>(W.w3b + (q - off_w3(D))) = h;
    *reinterpret_cast<float2*>(W.w3f + (q - off_w3(D))) = make_float2(bf16_lo(h), bf16_hi(h));
  } else {
    W.b3 = p.x;
  }
}

// Ring standardisation (the training set of the learned proposal), when th
// is non-null: z = max((log pi - max log pi) / tau, -8), tau = max(2, D), the
// target y = (z - mean z) / sd z; inputs standardised by the mean and sd of
// the rows above the clip (all rows if fewer than 2D + 2), moments taken about
// ring row 0; results into x, y (global) and *norm or stdz.  Then `steps` Adam steps.
struct MlpRing {
  const float* th;   // [rows][D]
  const float* lp;   // [rows]
  const int* rows;   // row count on the device, or null (then the kernel's R)
  MlpNorm* norm;     // the standardisation, or null
  double* stdz;      // mu[D], sd[D], tau, zmean, zsd, var_y, loss, ymax, or null
};

__global__ void __launch_bounds__(32 * kTrainWarps)
    mlp_train_kernel(float* p, float* m, float* v, int* step, float* x, float* y, int R_imm, float* loss, int D,
                     int steps, float lr, MlpRing ring) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  MlpTrainSmem& S = *reinterpret_cast<MlpTrainSmem*>(smem_raw);
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks(), c = (int)cluster.block_rank();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int P = mlp_nparams(D);
  const int R = ring.rows ? *ring.rows : R_imm;
  const int per = (R + C - 1) / C, r0 = min(c * per, R), r1 = min(r0 + per, R);
  // this thread's pair of parameters q, q + 1 (slice c of the pairs; further pairs of a
  // slice larger than the CTA, in clusters of fewer than 8, stay in global memory)
  const int n_pairs = (P + 1) / 2, slice = (n_pairs + C - 1) / C;
  const int q_end = 2 * min((c + 1) * slice, n_pairs), q_own = 2 * (c * slice + tid);
  auto load2 = [&](const float* a, int q) { return make_float2(a[q], q + 1 < P ? a[q + 1] : 0.f); };
  auto store2 = [&](float* a, int q, float2 w) {
    a[q] = w.x;
    if (q + 1 < P) a[q + 1] = w.y;
  };
  float2 own_p = make_float2(0.f, 0.f), own_m = own_p, own_v = own_p;
  if (q_own < q_end) {
    own_p = load2(p, q_own);
    own_m = load2(m, q_own);
    own_v = load2(v, q_own);
  }
  const int t0 = *step;
  for (int e = D * kLd + tid; e < 16 * kLd; e += blockDim.x) S.W.w1b[e] = __float2bfloat16_rn(0.f);
  for (int q = 2 * tid; q < P; q += 2 * blockDim.x) put_weights(S.W, D, q, load2(p, q));
  int n_tot = 0;
  if (ring.th) {
    const float tau = D > 2 ? (float)D : 2.f, inv_tau = 1.f / tau;
    constexpr int kStd = 32 * kStdWarps;
    const int rs = tid < kStd ? r0 + tid : r1;  // the rows of the summing threads
    float mx[1] = {-INFINITY};
    for (int r = rs; r < r1; r += kStd) {
      const float l = ring.lp[r];
      if (isfinite(l)) mx[0] = fmaxf(mx[0], l);
    }
    cluster_totals<1>(mx, S, cluster, true, n_tot);
    const float ymax = mx[0], cut = ymax - 8.f * tau;
    float ref[kMlpMaxD], mu[kMlpMaxD], sd[kMlpMaxD];
#pragma unroll
    for (int d = 0; d < kMlpMaxD; ++d) ref[d] = (R > 0 && d < D) ? ring.th[d] : 0.f;
    for (int pass = 0; pass < 2; ++pass) {  // pass 0: rows above the clip; pass 1: every finite row
      float acc[2 * kMlpMaxD + 1];
#pragma unroll
      for (int i = 0; i < 2 * kMlpMaxD + 1; ++i) acc[i] = 0.f;
      for (int r = rs; r < r1; r += kStd) {
        const float l = ring.lp[r];
        if (!isfinite(l) || (pass == 0 && l <= cut)) continue;
        acc[2 * kMlpMaxD] += 1.f;
#pragma unroll
        for (int d = 0; d < kMlpMaxD; ++d) {
          if (d >= D) break;
          const float cdev = ring.th[(size_t)r * D + d] - ref[d];
          acc[d] += cdev;
          acc[kMlpMaxD + d] += cdev * cdev;
        }
      }
      cluster_totals<2 * kMlpMaxD + 1>(acc, S, cluster, false, n_tot);
      const float cnt = acc[2 * kMlpMaxD];
#pragma unroll
      for (int d = 0; d < kMlpMaxD; ++d) {
        const float m1 = cnt > 0.f ? acc[d] / cnt : 0.f;
        const float m2 = cnt > 0.f ? acc[kMlpMaxD + d] / cnt : 0.f;
        mu[d] = ref[d] + m1;
        sd[d] = fmaxf(cnt > 1.f ? sqrtf(fmaxf(m2 - m1 * m1, 0.f)) : 1.f, 1e-6f);
      }
      if (cnt >= 2.f * D + 2.f) break;
    }
    auto z_of = [&](float l) { return isfinite(l) ? fmaxf((l - ymax) * inv_tau, -8.f) : -8.f; };
    float zs[2] = {0.f, 0.f};
    for (int r = rs; r < r1; r += kStd) {
      const float z = z_of(ring.lp[r]);
      zs[0] += z;
      zs[1] += z * z;
    }
    cluster_totals<2>(zs, S, cluster, false, n_tot);
    const float zmean = R > 0 ? zs[0] / (float)R : 0.f;
    const float zvar = R > 0 ? fmaxf(zs[1] / (float)R - zmean * zmean, 0.f) : 0.f;
    const float zsd = zvar > 1e-8f ? sqrtf(zvar) : 1.f, inv_zsd = 1.f / zsd;
    float inv_sd[kMlpMaxD];
#pragma unroll
    for (int d = 0; d < kMlpMaxD; ++d) inv_sd[d] = 1.f / sd[d];
    for (int r = r0 + tid; r < r1; r += blockDim.x) {
      y[r] = (z_of(ring.lp[r]) - zmean) * inv_zsd;
#pragma unroll
      for (int d = 0; d < kMlpMaxD; ++d) {
        if (d >= D) break;
        x[(size_t)r * D + d] = (ring.th[(size_t)r * D + d] - mu[d]) * inv_sd[d];
      }
    }
    if (c == 0 && tid == 0) {
      const float var_y = zvar > 1e-8f ? 1.f : 0.f;
      if (ring.norm) {
        MlpNorm& nm = *ring.norm;
#pragma unroll
        for (int d = 0; d < kMlpMaxD; ++d) {
          if (d >= D) break;
          nm.mu[d] = mu[d];
          nm.sd[d] = 1.0 / (double)inv_sd[d];
        }
        nm.ymax = ymax;
        nm.tau = tau;
        nm.zmean = zmean;
        nm.zsd = zsd;
        nm.rows = R;
        nm.var_y = var_y;
      }
      if (ring.stdz) {
#pragma unroll
        for (int d = 0; d < kMlpMaxD; ++d) {
          if (d >= D) break;
          ring.stdz[d] = mu[d];
          ring.stdz[D + d] = 1.0 / (double)inv_sd[d];
        }
        ring.stdz[2 * D] = tau;
        ring.stdz[2 * D + 1] = zmean;
        ring.stdz[2 * D + 2] = zsd;
        ring.stdz[2 * D + 3] = var_y;
        if (steps == 0) ring.stdz[2 * D + 4] = 0.0;
        ring.stdz[2 * D + 5] = ymax;
      }
    }
    __syncthreads();  // this CTA's rows of x, y written before it reads them back
  }
  if (steps == 0) {
    cluster.sync();  // no CTA exits while its totals may be read
    return;
  }
  const bool cached = r1 - r0 <= kTrainRows;  // one chunk: rows stay in shared memory
  const float beta1 = 0.9f, beta2 = 0.999f, eps = 1e-8f;
  const LaneTile lt;
  const int rt = 16 * warp;                                              // the warp's tile of the chunk
  // the gradient products: warps 0-7 take 32 x 16 of dW2 (units i from mt, o from nt), those with
  // mt = 0 also db2 of their units o; warps 8-15 eight units of [dW1; db1]
  const int mt = 32 * (warp & 1), nt = 16 * (warp >> 1 & 3), zc = 8 * (warp & 7);
  for (int it = 0; it < steps; ++it) {
    float acc[4][4], zacc[2][4];  // dW2 by 16 x 8 tiles (acc[0]: rows d < D dW1[d], row D db1); db2 in every row
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[0][e] = acc[1][e] = acc[2][e] = acc[3][e] = zacc[0][e] = zacc[1][e] = 0.f;
    float col_acc = 0.f, sc_acc = 0.f;  // dw3 of unit tid % 64 over tiles 2 (tid / 64), + 1; scalars likewise
    for (int base = r0; base < r1 || (base == r0 && r0 == r1); base += kTrainRows) {
      const int n = min(kTrainRows, r1 - base);
      if (!cached || it == 0) {
        for (int e = tid; e < kTrainRows; e += blockDim.x) S.ys[e] = e < n ? y[base + e] : 0.f;
        for (int e = tid; e < 16 * kTrainRows; e += blockDim.x) {
          const int d = e / kTrainRows, r = e % kTrainRows;
          S.xT[d * kLdT + r] =
              __float2bfloat16_rn(d < D ? (r < n ? x[(size_t)(base + r) * D + d] : 0.f) : (d == D ? 1.f : 0.f));
        }
        __syncthreads();
      }
      {
        const int ra = rt + g, rb = ra + 8;  // rows within the chunk
        uint32_t xp[4];
        ldsm4t(xp, S.xT + lt.lo2 * kLdT + rt + lt.hi2);
        WarpForward F;
        warp_forward(S.W, xp, F);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) stsm4(S.h1 + (rt + lt.lo) * kLd + 16 * kk + lt.hi, F.h1p[kk]);
        const float ea = ra < n ? F.s_lo - S.ys[ra] : 0.f, eb = rb < n ? F.s_hi - S.ys[rb] : 0.f;
        const float ga = 2.f * ea / (float)R, gb = 2.f * eb / (float)R;
        const float le = warp_sum(t == 0 ? ea * ea + eb * eb : 0.f), d3 = warp_sum(t == 0 ? ga + gb : 0.f);
        if (lane == 0) {
          S.sc[warp][0] = le;
          S.sc[warp][1] = d3;
        }
        // dw3 = sum_r h2_r ga_r (FP32 row signal): columns 8j + 2t + e summed over the lanes of equal t,
        // each exchange halving the columns that a lane keeps (the sums of a butterfly over g)
        float w3[8][2];
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
          for (int e = 0; e < 2; ++e) w3[j][e] = round_bf16(F.h2[j][e]) * ga + round_bf16(F.h2[j][2 + e]) * gb;
        int j3 = 0;
#pragma unroll
        for (int half = 4, bit = 1; half >= 1; half >>= 1, bit <<= 1) {
          const bool up = (g & bit) != 0;
          j3 += up ? half : 0;
#pragma unroll
          for (int j = 0; j < half; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const float give = up ? w3[j][e] : w3[j + half][e], keep = up ? w3[j + half][e] : w3[j][e];
              w3[j][e] = keep + __shfl_xor_sync(0xffffffffu, give, 4 * bit);
            }
        }
        *reinterpret_cast<float2*>(&S.col[warp][8 * j3 + 2 * t]) = make_float2(w3[0][0], w3[0][1]);
        uint32_t dz2[4][4], dz1[4][4];
        warp_backward(S.W, F, ga, gb, dz2, dz1);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          stsm4(S.dz2 + (rt + lt.lo) * kLd + 16 * kk + lt.hi, dz2[kk]);
          stsm4(S.dz1 + (rt + lt.lo) * kLd + 16 * kk + lt.hi, dz1[kk]);
        }
      }
      __syncthreads();
      {  // the tiles of two warps in turn, chunk by chunk
        const int w = 2 * (tid / kMlpH), e = tid % kMlpH;
        col_acc = (col_acc + S.col[w][e]) + S.col[w + 1][e];
        if (tid < kTrainWarps) {
          const int ws = tid & ~1;
          sc_acc = (sc_acc + S.sc[ws][tid & 1]) + S.sc[ws + 1][tid & 1];
        }
      }
      // dW2 += h1^T dz2, db2 += 1^T dz2, [dW1; db1] += [x^T; 1] dz1 over the chunk's rows
      if (warp < 8) {
#pragma unroll 4
        for (int kk = 0; kk < kTrainRows / 16; ++kk) {
          uint32_t a[4], a2[4], b[4];
          ldsm4t(b, S.dz2 + (16 * kk + lt.lo) * kLd + nt + lt.hi);
          ldsm4t(a, S.h1 + (16 * kk + lt.lo2) * kLd + mt + lt.hi2);
          ldsm4t(a2, S.h1 + (16 * kk + lt.lo2) * kLd + mt + 16 + lt.hi2);
          mma_bf16(acc[0], a[0], a[1], a[2], a[3], b[0], b[1]);
          mma_bf16(acc[1], a[0], a[1], a[2], a[3], b[2], b[3]);
          mma_bf16(acc[2], a2[0], a2[1], a2[2], a2[3], b[0], b[1]);
          mma_bf16(acc[3], a2[0], a2[1], a2[2], a2[3], b[2], b[3]);
          if (mt == 0) {
            constexpr uint32_t kOnes = 0x3f803f80u;
            mma_bf16(zacc[0], kOnes, kOnes, kOnes, kOnes, b[0], b[1]);
            mma_bf16(zacc[1], kOnes, kOnes, kOnes, kOnes, b[2], b[3]);
          }
        }
      } else {
#pragma unroll 4
        for (int kk = 0; kk < kTrainRows / 16; ++kk) {
          uint32_t xa[4], z0, z1;
          ldsm4(xa, S.xT + lt.lo * kLdT + 16 * kk + lt.hi);
          ldsm2t(z0, z1, S.dz1 + (16 * kk + lt.lo) * kLd + zc);
          mma_bf16(acc[0], xa[0], xa[1], xa[2], xa[3], z0, z1);
        }
      }
      if (r0 == r1) break;
      if (!cached) __syncthreads();  // staging and rows free for the next chunk
    }
    // the CTA's partial gradient into gp
    if (warp < 8) {
      float* gW2 = S.gp + off_W2(D);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int i0 = mt + 16 * (j >> 1) + g, o = nt + 8 * (j & 1) + 2 * t;
        *reinterpret_cast<float2*>(gW2 + i0 * kMlpH + o) = make_float2(acc[j][0], acc[j][1]);
        *reinterpret_cast<float2*>(gW2 + (i0 + 8) * kMlpH + o) = make_float2(acc[j][2], acc[j][3]);
      }
      if (mt == 0 && g < 2)  // every row of zacc holds db2
        *reinterpret_cast<float2*>(S.gp + off_b2(D) + nt + 8 * g + 2 * t) =
            g ? make_float2(zacc[1][0], zacc[1][1]) : make_float2(zacc[0][0], zacc[0][1]);
    } else {  // rows g (c0, c1) and g + 8 (c2, c3) of the [x^T; 1] products
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int row = g + 8 * h;
        float* to = row < D ? S.gp + row * kMlpH : S.gp + off_b1(D);
        if (row <= D) *reinterpret_cast<float2*>(to + zc + 2 * t) = make_float2(acc[0][2 * h], acc[0][2 * h + 1]);
      }
    }
    S.pairs[tid / kMlpH][tid % kMlpH] = col_acc;
    if (tid < kTrainWarps) S.psc[tid >> 1][tid & 1] = sc_acc;
    __syncthreads();
    if (tid < kMlpH + 2) {  // dw3, then the sum of e^2 (after b3's gradient) and db3
      float s = 0.f;
      for (int w = 0; w < kTrainWarps / 2; ++w) s += tid < kMlpH ? S.pairs[w][tid] : S.psc[w][tid - kMlpH];
      S.gp[tid < kMlpH ? off_w3(D) + tid : (tid == kMlpH ? P : off_b3(D))] = s;
    }
    auto arrival = cluster.barrier_arrive();  // every CTA's partial gradient complete
    const int tstep = t0 + it + 1;
    float bc1 = 1.f, bc2 = 1.f;
    if (q_own < q_end) {  // the few warps that step parameters, while the others' gradients arrive
      bc1 = 1.f - powf(beta1, (float)tstep);
      bc2 = 1.f - powf(beta2, (float)tstep);
    }
    cluster.barrier_wait(std::move(arrival));
    auto adam = [&](float pq, float sum, float& mq, float& vq) {
      // fused multiply-adds written out: the compiler's choice of them moves the last bit
      const float mn = __fmaf_rn(1.f - beta1, sum, __fmul_rn(beta1, mq));
      const float vn = __fmaf_rn(__fmul_rn(1.f - beta2, sum), sum, __fmul_rn(beta2, vq));
      mq = mn;
      vq = vn;
      return pq - lr * (mn / bc1) / (sqrtf(vn / bc2) + eps);
    };
    auto update = [&](int q, float2& pq, float2& mq, float2& vq) {
      float2 part[kMaxCluster];  // every rank's partial in flight at once, summed in rank order
#pragma unroll
      for (int r = 0; r < kMaxCluster; ++r)
        part[r] = r < C ? *reinterpret_cast<const float2*>(cluster.map_shared_rank(S.gp + q, r)) : make_float2(0.f, 0.f);
      float sx = 0.f, sy = 0.f;
#pragma unroll
      for (int r = 0; r < kMaxCluster; ++r) {
        sx += part[r].x;
        sy += part[r].y;
      }
      pq.x = adam(pq.x, sx, mq.x, vq.x);
      if (q + 1 < P) pq.y = adam(pq.y, sy, mq.y, vq.y);
      if (q == off_b3(D) && it == steps - 1) {  // gp[q + 1] is the loss sum
        const float l = R > 0 ? sy / (float)R : 0.f;
        if (loss) *loss = l;
        if (ring.stdz) ring.stdz[2 * D + 4] = l;
      }
      for (int r = 0; r < C; ++r) put_weights(*cluster.map_shared_rank(&S.W, r), D, q, pq);
    };
    if (q_own < q_end) update(q_own, own_p, own_m, own_v);
    for (int q = q_own + 2 * (int)blockDim.x; q < q_end; q += 2 * blockDim.x) {
      float2 pq = load2(p, q), mq = load2(m, q), vq = load2(v, q);
      update(q, pq, mq, vq);
      store2(p, q, pq);
      store2(m, q, mq);
      store2(v, q, vq);
    }
    cluster.sync();  // every operand copy updated; partial gradients free again
  }
  if (q_own < q_end) {
    store2(p, q_own, own_p);
    store2(m, q_own, own_m);
    store2(v, q_own, own_v);
  }
  if (c == 0 && tid == 0) *step = t0 + steps;
}

// s and ds/dx of a warp's rows g and g+8: lane (g, t) returns dx of
// coordinates 2t and 2t+1 (rows g: dx_lo, g+8: dx_hi).
__device__ __forceinline__ void warp_input_grad(const MlpSmemWeights& W, const float* xa, const float* xb,
                                                WarpForward& F, float (&dx_lo)[2], float (&dx_hi)[2]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const uint32_t xp[4] = {pack_bf16(xa[0], xa[1]), pack_bf16(xb[0], xb[1]), pack_bf16(xa[2], xa[3]),
                          pack_bf16(xb[2], xb[3])};
  warp_forward(W, xp, F);
  uint32_t dz2[4][4], dz1[4][4];
  warp_backward(W, F, 1.f, 1.f, dz2, dz1);
  // dx = dz1 W1^T: k over the hidden units, n over the input coordinates (padded to 8)
  float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int kk = 0; kk < 4; ++kk) {
    const bf16* w = W.w1b + g * kLd + 16 * kk + 2 * t;
    mma_bf16(c, dz1[kk][0], dz1[kk][1], dz1[kk][2], dz1[kk][3], ld32(w), ld32(w + 8));
  }
  dx_lo[0] = c[0];
  dx_lo[1] = c[1];
  dx_hi[0] = c[2];
  dx_hi[1] = c[3];
}

// s(x) and ds/dx of R rows.
__global__ void __launch_bounds__(32 * kMlpWarps)
    mlp_input_grad_kernel(const float* __restrict__ p, int D, const float* __restrict__ x, int R,
                          float* __restrict__ s_out, float* __restrict__ dx) {
  __shared__ MlpSmemWeights W;
  load_weights(W, p, D);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int ra = blockIdx.x * kRowsCta + warp * 16 + g, rb = ra + 8;
  const bool va = ra < R, vb = rb < R;
  float xa[4], xb[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int k = 2 * t + (e & 1) + (e >> 1) * 8;
    xa[e] = (va && k < D) ? x[(size_t)ra * D + k] : 0.f;
    xb[e] = (vb && k < D) ? x[(size_t)rb * D + k] : 0.f;
  }
  WarpForward F;
  float dlo[2], dhi[2];
  warp_input_grad(W, xa, xb, F, dlo, dhi);
  if (t == 0) {
    if (va && s_out) s_out[ra] = F.s_lo;
    if (vb && s_out) s_out[rb] = F.s_hi;
  }
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int d = 2 * t + e;
    if (d < D) {
      if (va) dx[(size_t)ra * D + d] = dlo[e];
      if (vb) dx[(size_t)rb * D + d] = dhi[e];
    }
  }
}

// ---------------------------------------------------------------------------
// the learned proposal inside the sampler (dataset 0)
// ---------------------------------------------------------------------------

// Xavier-uniform weights and zero biases from the random stream (tag MLP_INIT);
// Adam moments and step cleared.
__global__ void mlp_init_kernel(MlpDev M, int D, uint64_t seed) {
  const int P = mlp_nparams(D);
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q == 0) *M.step = 0;
  if (q >= P) return;
  const float u = 2.f * uniform23<float>(philox4x32_10(make_uint4((uint32_t)q, 0u, 0u, TAG_MLP_INIT),
                                                       seed_key(seed)).x) - 1.f;
  float a = 0.f;
  if (q < off_b1(D))
    a = sqrtf(6.f / (float)(D + kMlpH));
  else if (q >= off_W2(D) && q < off_b2(D))
    a = sqrtf(6.f / (float)(2 * kMlpH));
  else if (q >= off_w3(D) && q < off_b3(D))
    a = sqrtf(6.f / (float)(kMlpH + 1));
  M.p[q] = a * u;
  M.p_use[q] = a * u;
  M.m[q] = 0.f;
  M.v[q] = 0.f;
}

// (theta_k, log pi^(theta_k)) of this iteration's proposals into ring slot (k-1) mod W.
__global__ void mlp_append_kernel(OuterParams P) {
  const DSDev& S = P.ds[0];
  const int k = *P.k_done + 1, N = S.N, D = P.D;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const size_t row = (size_t)((k - 1) % P.mlp.W) * N + i;
  for (int d = 0; d < D; ++d) P.mlp.ring_th[row * D + d] = (float)S.thB[(size_t)d * N + i];
  P.mlp.ring_lp[row] = (float)(S.lpB[i] + S.llB[i]);
  if (i == 0) *P.mlp.ring_rows = min(k, P.mlp.W) * N;
}

// The trained state becomes the one the proposal reads.
__global__ void mlp_publish_kernel(MlpDev M, int n_par) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < n_par) M.p_use[q] = M.p[q];
  if (q == 0) {
    *M.norm_use = *M.norm;
    *M.loss_use = *M.loss;
  }
}

// Score of the surrogate at the parents theta_{k-1}: through the input and
// target standardisations, d log pi^ / d theta_d = tau zsd (ds/dx)_d / sd_d.
// Decides whether iteration k proposes with it: from k = 3 on, while the
// published network explains half the variance of its targets and the
// population covariance has a usable Cholesky factor.
__global__ void __launch_bounds__(32 * kMlpWarps) mlp_score_kernel(OuterParams P) {
  __shared__ MlpSmemWeights W;
  const DSDev& S = P.ds[0];
  const int k = *P.k_done + 1, N = S.N, D = P.D;
  const MlpNorm& nm = *P.mlp.norm_use;
  const float loss = *P.mlp.loss_use;
  const bool use = k >= 3 && isfinite(loss) && nm.var_y > 0.f && loss < 0.5f * nm.var_y && S.cur->pop_ok;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    S.cur->mlp_used = use ? 1 : 0;
    S.cur->mlp_loss = (double)loss;
  }
  if (!use) return;
  load_weights(W, P.mlp.p_use, D);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int ra = blockIdx.x * kRowsCta + warp * 16 + g, rb = ra + 8;
  const bool va = ra < N, vb = rb < N;
  float xa[4], xb[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int d = 2 * t + (e & 1) + (e >> 1) * 8;
    xa[e] = (va && d < D) ? (float)((S.thA[(size_t)d * N + ra] - nm.mu[d]) / nm.sd[d]) : 0.f;
    xb[e] = (vb && d < D) ? (float)((S.thA[(size_t)d * N + rb] - nm.mu[d]) / nm.sd[d]) : 0.f;
  }
  WarpForward F;
  float dlo[2], dhi[2];
  warp_input_grad(W, xa, xb, F, dlo, dhi);
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int d = 2 * t + e;
    if (d >= D) continue;
    const double scale = nm.tau * nm.zsd / nm.sd[d];
    if (va) P.mlp.score[(size_t)d * N + ra] = scale * dlo[e];
    if (vb) P.mlp.score[(size_t)d * N + rb] = scale * dhi[e];
  }
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
int mlp_param_count(int D) { return mlp_nparams(D); }
int mlp_grad_ctas(int R) { return (R + kRowsGrad - 1) / kRowsGrad; }

// One gradient (and optionally Adam) step over R rows (R_dev, when given, holds
// the row count; R bounds it and sizes the grid).
cudaError_t mlp_step_launch(float* p, int D, const float* x, const float* y, int R, const int* R_dev,
                            float* part, float* grad, float* loss, int adam, float* m, float* v, int* step,
                            float lr, cudaStream_t s) {
  const size_t smem = sizeof(MlpGradSmem);
  cudaError_t e = cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  mlp_grad_kernel<<<mlp_grad_ctas(R), 32 * kGradWarps, smem, s>>>(p, D, x, y, R, R_dev, part,
                                                                  adam ? step : nullptr);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int P = mlp_nparams(D);
  mlp_reduce_kernel<<<(P + 1 + 127) / 128, 128, 0, s>>>(p, D, part, R, R_dev, grad, loss, adam, m, v, step,
                                                         lr);
  return cudaGetLastError();
}

cudaError_t mlp_train_footprint(int* ctas, int* threads, int* regs, size_t* smem) {
  cudaFuncAttributes a{};
  const cudaError_t e = cudaFuncGetAttributes(&a, mlp_train_kernel);
  if (e != cudaSuccess) return e;
  *ctas = mlp_train_cluster_size();
  *threads = 32 * kTrainWarps;
  *regs = a.numRegs;
  *smem = sizeof(MlpTrainSmem) + a.sharedSizeBytes;
  return cudaSuccess;
}

// Largest cluster (16, 8, 4, 2 or 1 CTAs) that the device can co-schedule with
// this kernel's shared memory.
int mlp_train_cluster_size() {
  static int cached = 0;
  if (cached) return cached;
  const size_t smem = sizeof(MlpTrainSmem);
  if (cudaFuncSetAttribute(mlp_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
          cudaSuccess ||
      cudaFuncSetAttribute(mlp_train_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
    return 0;
  for (int C = 16; C >= 1; C >>= 1) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(32 * kTrainWarps);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, mlp_train_kernel, &cfg) == cudaSuccess && n > 0) {
      cached = C;
      return C;
    }
    cudaGetLastError();
  }
  return 0;
}

static cudaError_t train_launch(float* p, float* m, float* v, int* step, float* x, float* y, int R, float* loss,
                                int D, int steps, float lr, const MlpRing& ring, cudaStream_t s) {
  const int C = mlp_train_cluster_size();
  if (C < 1) return cudaErrorInvalidConfiguration;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(C);
  cfg.blockDim = dim3(32 * kTrainWarps);
  cfg.dynamicSmemBytes = sizeof(MlpTrainSmem);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, mlp_train_kernel, p, m, v, step, x, y, R, loss, D, steps, lr, ring);
}

// Adam steps on the training set (x, y) of R rows.
cudaError_t mlp_train_steps_launch(float* p, float* m, float* v, int* step, float* x, float* y, int R, float* loss,
                                   int D, int steps, float lr, cudaStream_t s) {
  return train_launch(p, m, v, step, x, y, R, loss, D, steps, lr, MlpRing{}, s);
}

// The training call on caller buffers: the ring (th, lp) of R rows is standardised
// into x, y and stdz (mu[D], sd[D], tau, zmean, zsd, var_y, loss, ymax), then `steps`
// Adam steps continue (p, m, v, *step); the sampler's own kernel and cluster shape.
cudaError_t mlp_train_ring_launch(float* p, float* m, float* v, int* step, const float* th, const float* lp, int R,
                                  float* x, float* y, double* stdz, int D, int steps, float lr, cudaStream_t s) {
  return train_launch(p, m, v, step, x, y, R, nullptr, D, steps, lr, MlpRing{th, lp, nullptr, nullptr, stdz}, s);
}

cudaError_t mlp_init_launch(const MlpDev& M, int D, uint64_t seed, cudaStream_t s) {
  const int P = mlp_nparams(D);
  mlp_init_kernel<<<(P + 255) / 256, 256, 0, s>>>(M, D, seed);
  return cudaGetLastError();
}

// Store this iteration's rows (before resampling moves the population).
cudaError_t mlp_append_launch(const OuterParams& P, int N, cudaStream_t s) {
  mlp_append_kernel<<<(N + 127) / 128, 128, 0, s>>>(P);
  return cudaGetLastError();
}

// Standardise the ring and take `steps` Adam steps on it: one cluster launch.
cudaError_t mlp_train_launch(const OuterParams& P, int steps, float lr, cudaStream_t s) {
  const MlpDev& M = P.mlp;
  return train_launch(M.p, M.m, M.v, M.step, M.xs, M.ys, M.W * P.ds_N0, M.loss, P.D, steps, lr,
                      MlpRing{M.ring_th, M.ring_lp, M.ring_rows, M.norm, nullptr}, s);
}

cudaError_t mlp_publish_launch(const OuterParams& P, cudaStream_t s) {
  const int n_par = mlp_nparams(P.D);
  mlp_publish_kernel<<<(n_par + 255) / 256, 256, 0, s>>>(P.mlp, n_par);
  return cudaGetLastError();
}

cudaError_t mlp_score_launch(const OuterParams& P, int N, cudaStream_t s) {
  mlp_score_kernel<<<(N + kRowsCta - 1) / kRowsCta, 32 * kMlpWarps, 0, s>>>(P);
  return cudaGetLastError();
}

cudaError_t mlp_input_grad_launch(const float* p, int D, const float* x, int R, float* s_out, float* dx,
                                  cudaStream_t s) {
  mlp_input_grad_kernel<<<(R + kRowsCta - 1) / kRowsCta, 32 * kMlpWarps, 0, s>>>(p, D, x, R, s_out, dx);
  return cudaGetLastError();
}

}  // namespace smc2
