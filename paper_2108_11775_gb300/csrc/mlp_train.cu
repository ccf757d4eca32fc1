// Training step of the surrogate network (39 -> 128 -> 128 -> 128 -> 3, see
// mlp.cu) in two launches: forward, backward and weight gradients in one kernel,
// then the sum of its partial gradients with Adam (or into gW, gb) and the loss.
//
// A training batch is small (some thousand pairs, under 1 GFLOP), so what
// counts is the length of the chain a warp goes through and the passes over
// memory between launches, not the arithmetic.  A cluster of two blocks takes
// 64 samples, 32 a block; a block's sixteen warps are 2 row tiles of 16 x 8
// groups of 16 columns, so a layer is 16 mma.sync (m16n8k16, BF16 x BF16 -> FP32)
// a warp.  A layer's output goes to shared memory as BF16, both as
// the next layer's A operand and as an operand of the weight gradients, and
// pre-activations stay in the registers of the lanes that need them on the way
// back.  W2 and W3 are in shared memory once, read as they lie forwards and
// transposed (ldmatrix.trans) backwards.
//
// The weight and bias gradients are [dW_l | db_l] = dZ_l^T [a_{l-1} | 1] over
// the 64 samples (a column of ones behind the activations).  Each block of the
// pair takes 64 of the 128 output units, for which every block writes its
// activations into the other's shared memory too, and its dZ as far as the
// other takes them.  The partial sums of 64 samples go to memory and are added
// in sample order.
//
// Measured (us a step, before: seven launches with the activations in memory and
// one warp per 16 samples; eight warps a block with 32 columns each; now): 256
// pairs 133 / 40 / 33, 4096 pairs 128 / 37 / 26, 16,384 pairs 261 / 109 / 86.
// Of the 26, 19 are this kernel, whose bound is latency: 2500 instructions a warp
// in fourteen dependent stages on one block per SM.
#include <type_traits>

#include "fast_tile.cuh"
#include "kernels.cuh"
#include "mlp_common.cuh"

namespace pdmp {

namespace {

constexpr int kH = 128, kEnc = 39;
constexpr int kTrThreads = 512;               // 16 warps: 2 row tiles x 8 column groups of 16
constexpr int kStepThreads = 256;
constexpr int kTrRows = 64;                    // samples of a cluster (one part of the gradient)
constexpr int kTrOwn = kTrRows / 2;            // samples of a block
constexpr int kRow = 136;                      // row of W2, W3, a_l, dZ_l: 272 bytes (ldmatrix without conflicts)
constexpr int kRow0 = 40;                      // row of a_0: the encoding and its one
constexpr int kRowY = 24;                      // row of dY (16 columns used)
constexpr int kPart = kMlpTrainPart;
constexpr int kRowE = 44;                      // FP32 rows of the encoding and of W1

struct TrainSmem {
  uint16_t W2[kH * kRow], W3[kH * kRow];       // [out][in]
  uint16_t W4[8 * kRow];                       // rows 3 .. 7 zero
  uint16_t a[3][kTrRows * kRow];               // a_1, a_2, a_3: [sample][unit], a one in column 128, zeros behind
  uint16_t dz[3][kTrRows * kRow];              // dZ_1, dZ_2, dZ_3
  uint16_t a0[kTrRows * kRow0];
  uint16_t dy[kTrRows * kRowY];
  float W1[kH * kRowE];
  float enc[kTrOwn * kRowE];
  float W4f[3 * kH];
  float b[3 * kH + 4];
  float dyf[kTrOwn * 4];
};
static_assert(sizeof(TrainSmem) <= 227 * 1024, "shared memory of one block");

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const uint16_t* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p))
               : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const uint16_t* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p))
               : "memory");
}
__device__ __forceinline__ void ldsm2t(uint32_t& r0, uint32_t& r1, const uint16_t* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];"
               : "=r"(r0), "=r"(r1)
               : "r"((uint32_t)__cvta_generic_to_shared(p))
               : "memory");
}

// A word (two BF16 of a row) into this block's array and the other's.
__device__ __forceinline__ void put_both(uint16_t* p, int other, uint32_t v) {
  *reinterpret_cast<uint32_t*>(p) = v;
  cluster_store(cluster_addr(p, other), v);
}

// The warp's 16 x 16 of A W^T (FORWARD, W[n][k]) or A W (W[k][n]): A's 16 rows
// from `rows`, columns n0 .. n0 + 15 of the result.
template <bool FORWARD>
__device__ __forceinline__ void dense16x16(const uint16_t* rows, const uint16_t* W, int n0, int lane,
                                           float (&acc)[2][4]) {
#pragma unroll
  for (int j = 0; j < 2; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.0f;
  const uint16_t* pa = rows + (lane & 15) * kRow + (lane >> 4) * 8;
  // forward: matrices (columns 0: k 0, k 8), (columns 8: k 0, k 8), rows n
  // backward: the same matrices, rows k, transposed on the way
  const uint16_t* pb = FORWARD ? W + (n0 + (lane & 7) + (lane >> 4) * 8) * kRow + (lane >> 3 & 1) * 8
                               : W + (lane & 15) * kRow + n0 + (lane >> 4) * 8;
#pragma unroll
  for (int kk = 0; kk < 8; ++kk) {
    uint32_t af[4], b[4];
    ldsm4(af, pa + 16 * kk);
    if (FORWARD) ldsm4(b, pb + 16 * kk);
    else ldsm4t(b, pb + 16 * kk * kRow);
    mma16816(acc[0], af, b[0], b[1]);
    mma16816(acc[1], af, b[2], b[3]);
  }
}

// [dW | db] of one 16-unit m tile and NT n tiles from column 8 nt0 on, over the 64
// samples: dz (A, [sample][unit] from unit m0) and a (B, [sample][unit], row
// stride ra), into the part's rows of O units x I inputs.  c == I: the ones.
template <int NT, int O, int I>
__device__ __forceinline__ void grad_tiles64(const uint16_t* dz, int rz, int m0, const uint16_t* a, int ra, int nt0,
                                             int lane, float* __restrict__ W, float* __restrict__ b) {
  const int g = lane >> 2, t = lane & 3;
  float acc[NT][4];
#pragma unroll
  for (int j = 0; j < NT; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.0f;
  const uint16_t* pa = dz + ((lane & 7) + (lane >> 4) * 8) * rz + m0 + (lane >> 3 & 1) * 8;
  const uint16_t* pb = a + (lane & 15) * ra + 8 * nt0 + (lane >> 4) * 8;
#pragma unroll
  for (int kk = 0; kk < kTrRows / 16; ++kk) {
    uint32_t af[4];
    ldsm4t(af, pa + 16 * kk * rz);
#pragma unroll
    for (int j = 0; j + 1 < NT; j += 2) {
      uint32_t bf[4];
      ldsm4t(bf, pb + 16 * kk * ra + 8 * j);
      mma16816(acc[j], af, bf[0], bf[1]);
      mma16816(acc[j + 1], af, bf[2], bf[3]);
    }
    if (NT & 1) {
      uint32_t b0, b1;
      ldsm2t(b0, b1, a + (16 * kk + (lane & 15)) * ra + 8 * (nt0 + NT - 1));
      mma16816(acc[NT - 1], af, b0, b1);
    }
  }
#pragma unroll
  for (int j = 0; j < NT; ++j)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int o = m0 + g + 8 * h, c = 8 * (nt0 + j) + 2 * t;
      const float v0 = acc[j][2 * h], v1 = acc[j][2 * h + 1];
      if (o >= O) continue;
      if (I % 2 == 0) {
        if (c < I) *reinterpret_cast<float2*>(W + o * I + c) = make_float2(v0, v1);
        else if (c == I) b[o] = v0;
      } else {
        if (c < I) W[o * I + c] = v0;
        if (c + 1 < I) W[o * I + c + 1] = v1;
        else if (c + 1 == I) b[o] = v1;
      }
    }
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kTrThreads, 1)
k_mlp_train(MlpArgs a, const float* __restrict__ x0, const float* __restrict__ xT, int B, int parts,
            float* __restrict__ err, float* __restrict__ part) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TrainSmem* s = reinterpret_cast<TrainSmem*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const int crank = (int)(blockIdx.x & 1), other = crank ^ 1;
  const int rt = warp >> 3, n0 = 16 * (warp & 7);       // the warp's row tile and first column
  const int half0 = 64 * crank;                         // first of the output units whose gradients this block takes

  // ---- weights: all loads first, W2 and W3 arrive while the first layer runs
  const uint32_t* W1w = reinterpret_cast<const uint32_t*>(a.W1);
  constexpr int n1 = kH * kEnc / 2, per1 = (n1 + kTrThreads - 1) / kTrThreads;
  uint32_t w1[per1];
#pragma unroll
  for (int q = 0; q < per1; ++q) w1[q] = tid + q * kTrThreads < n1 ? W1w[tid + q * kTrThreads] : 0u;
  const uint32_t w4 = tid < 3 * kH / 2 ? reinterpret_cast<const uint32_t*>(a.W4)[tid] : 0u;
  const float bv = tid < 3 * kH + 3 ? a.b1[tid] : 0.0f;   // b1, b2, b3, b4
  static_assert(kH * kEnc % 8 == 0, "W2 and W3 start on 16-byte boundaries, as the weights do");
#pragma unroll
  for (int q = 0; q < kH * kH / 8 / kTrThreads; ++q) {
    const int i = tid + q * kTrThreads, r = i / (kH / 8), c = 8 * (i % (kH / 8));
    cp_async16(s->W2 + r * kRow + c, a.W2 + r * kH + c);
    cp_async16(s->W3 + r * kRow + c, a.W3 + r * kH + c);
  }
  cp_async_commit();
#pragma unroll
  for (int q = 0; q < per1; ++q) {
    const int i = 2 * (tid + q * kTrThreads);
    if (i < kH * kEnc) {
      s->W1[i / kEnc * kRowE + i % kEnc] = __uint_as_float(w1[q] << 16);
      s->W1[(i + 1) / kEnc * kRowE + (i + 1) % kEnc] = __uint_as_float(w1[q] & 0xffff0000u);
    }
  }
  if (tid < kH) s->W1[tid * kRowE + kEnc] = 0.0f;       // the pad that a float4 takes along
  if (tid < kTrOwn) s->enc[tid * kRowE + kEnc] = 0.0f;
  {
    const int r = tid / (kH / 2), c = 2 * (tid % (kH / 2));   // 8 rows x 64 words
    *reinterpret_cast<uint32_t*>(s->W4 + r * kRow + c) = w4;
    if (r < 3) {
      s->W4f[r * kH + c] = __uint_as_float(w4 << 16);
      s->W4f[r * kH + c + 1] = __uint_as_float(w4 & 0xffff0000u);
    }
  }
  static_assert(kTrThreads == 8 * kH / 2, "a word of W4 a thread");
  if (tid < 3 * kH + 3) s->b[tid] = bv;
  for (int i = tid; i < kTrRows * kRowY; i += kTrThreads) s->dy[i] = 0;
  cluster_arrive();   // waited for before the first write to the other block

  const float inv = 2.0f / (3.0f * (float)B);
  bool first = true;
  for (int p = (int)(blockIdx.x >> 1); p < parts; p += (int)(gridDim.x >> 1)) {
    const int64_t base = (int64_t)p * kTrRows;
    const int64_t own = base + crank * kTrOwn;          // this block's first sample
    // ---- the encoding: of all 64 samples as BF16 (an operand of dW_1), of the block's own in FP32
    {
      static_assert(kTrThreads == 8 * kTrRows, "eight threads a sample, of different warps: an octave each, the rest");
      const int r = tid & (kTrRows - 1), q = tid / kTrRows;
      const int64_t n = base + r;
      float x[3] = {0.0f, 0.0f, 0.0f};
      if (n < B)
#pragma unroll
        for (int j = 0; j < 3; ++j) x[j] = x0[n * 3 + j];
      MlpEncIn in;
      mlp_enc_prepare(x, a.lo, a.in_scale, in);
      const bool mine = (r >> 5) == crank;
      float* e = s->enc + (r & (kTrOwn - 1)) * kRowE;
#pragma unroll
      for (int f = 0; f < kEnc; ++f)
        if ((f < 3 ? 6 : (f - 3) / 6) == q) {
          const float v = mlp_enc_feature<false>(f, in);
          s->a0[r * kRow0 + f] = n < B ? bf16_bits(v) : (uint16_t)0;
          if (mine) e[f] = v;
        }
      if (q == 7) {   // the ones behind the encoding and behind a_1 .. a_3 (column 128), BF16 1.0
        s->a0[r * kRow0 + kEnc] = n < B ? 0x3f80 : 0;
#pragma unroll
        for (int l = 0; l < 3; ++l)
          *reinterpret_cast<uint4*>(&s->a[l][r * kRow + kH]) = make_uint4(n < B ? 0x3f80u : 0u, 0u, 0u, 0u);
      }
    }
    __syncthreads();
    const int rr[2] = {rt * 16 + g, rt * 16 + g + 8};   // the lane's rows among the block's own
    const bool in_b[2] = {own + rr[0] < B, own + rr[1] < B};
    float z[3][2][4];
    // ---- layer 1 (FP32)
    {
      float acc[2][4];
#pragma unroll
      for (int j = 0; j < 2; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.0f;
      const float* e0 = s->enc + rr[0] * kRowE;
      const float* e1 = s->enc + rr[1] * kRowE;
#pragma unroll 2
      for (int i = 0; i < kRowE - 4; i += 4) {
        float u0[4], u1[4];
        *reinterpret_cast<float4*>(u0) = *reinterpret_cast<const float4*>(e0 + i);
        *reinterpret_cast<float4*>(u1) = *reinterpret_cast<const float4*>(e1 + i);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          float wa[4], wb[4];
          const float* w = s->W1 + (n0 + 8 * j + 2 * t) * kRowE + i;
          *reinterpret_cast<float4*>(wa) = *reinterpret_cast<const float4*>(w);
          *reinterpret_cast<float4*>(wb) = *reinterpret_cast<const float4*>(w + kRowE);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            acc[j][0] = fmaf(wa[q], u0[q], acc[j][0]);
            acc[j][1] = fmaf(wb[q], u0[q], acc[j][1]);
            acc[j][2] = fmaf(wa[q], u1[q], acc[j][2]);
            acc[j][3] = fmaf(wb[q], u1[q], acc[j][3]);
          }
        }
      }
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) z[0][j][q] = acc[j][q];
    }
    if (first) {
      cp_async_wait_all();   // the barrier below publishes W2 and W3
      cluster_wait();
      first = false;
    }
    // bias + SiLU of layer l + 1: the pre-activations stay in z, the activations go to both blocks
    auto activate = [&](auto lc) {
      constexpr int l = decltype(lc)::value;
      const float* bias = s->b + l * kH;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int c = n0 + 8 * j + 2 * t;
#pragma unroll
        for (int q = 0; q < 4; ++q) z[l][j][q] += bias[c + (q & 1)];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const uint32_t v = in_b[h] ? pack_bf16(silu_f(z[l][j][2 * h]), silu_f(z[l][j][2 * h + 1])) : 0u;
          put_both(s->a[l] + (crank * kTrOwn + rr[h]) * kRow + c, other, v);
        }
      }
    };
    const int row0 = crank * kTrOwn + rt * 16;          // the warp's rows among the 64
    activate(std::integral_constant<int, 0>());
    __syncthreads();
    dense16x16<true>(s->a[0] + row0 * kRow, s->W2, n0, lane, z[1]);
    activate(std::integral_constant<int, 1>());
    __syncthreads();
    dense16x16<true>(s->a[1] + row0 * kRow, s->W3, n0, lane, z[2]);
    activate(std::integral_constant<int, 2>());
    __syncthreads();
    // ---- output layer, its error and dY: one warp a row tile
    if ((warp & 7) == 0) {
      float o[4] = {0.0f, 0.0f, 0.0f, 0.0f};
      const uint16_t* pa = s->a[2] + (row0 + (lane & 15)) * kRow + (lane >> 4) * 8;
      const uint16_t* pb = s->W4 + g * kRow + 2 * t;
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) {
        uint32_t af[4];
        ldsm4(af, pa + 16 * kk);
        mma16816(o, af, *reinterpret_cast<const uint32_t*>(pb + 16 * kk),
                 *reinterpret_cast<const uint32_t*>(pb + 16 * kk + 8));
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int64_t n = own + rr[h];
        float q2 = 0.0f, d[2] = {0.0f, 0.0f};
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int c = 2 * t + q;
          if (c < 3 && n < B) {
            const float scale = c == 0 ? a.out_scale[0] : (c == 1 ? a.out_scale[1] : a.out_scale[2]);
            const float tgt = (xT[n * 3 + c] - x0[n * 3 + c]) / scale;
            const float r = o[2 * h + q] + s->b[3 * kH + c] - tgt;
            d[q] = inv * r;
            q2 += r * r;
          }
        }
        if (t < 2) {
          s->dyf[rr[h] * 4 + 2 * t] = d[0];
          s->dyf[rr[h] * 4 + 2 * t + 1] = d[1];
          put_both(s->dy + (crank * kTrOwn + rr[h]) * kRowY + 2 * t, other, pack_bf16(d[0], d[1]));
        }
        q2 += __shfl_xor_sync(0xffffffffu, q2, 1);
        if (t == 0 && n < B) err[n] = q2;
      }
    }
    __syncthreads();
    // ---- backward: dZ_l = dA_l silu'(z_l), dA_{l-1} = dZ_l W_l
    float acc[2][4];
    {
      const float* d0 = s->dyf + rr[0] * 4;
      const float* d1 = s->dyf + rr[1] * 4;
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int c = n0 + 8 * j + 2 * t + q;
          acc[j][q] = d0[0] * s->W4f[c] + d0[1] * s->W4f[kH + c] + d0[2] * s->W4f[2 * kH + c];
          acc[j][2 + q] = d1[0] * s->W4f[c] + d1[1] * s->W4f[kH + c] + d1[2] * s->W4f[2 * kH + c];
        }
    }
    auto back = [&](auto lc) {
      constexpr int l = decltype(lc)::value;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int c = n0 + 8 * j + 2 * t;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float v0 = acc[j][2 * h] * silu_grad_f(z[l][j][2 * h]);
          const float v1 = acc[j][2 * h + 1] * silu_grad_f(z[l][j][2 * h + 1]);
          const uint32_t v = in_b[h] ? pack_bf16(v0, v1) : 0u;
          uint16_t* d = s->dz[l] + (crank * kTrOwn + rr[h]) * kRow + c;
          *reinterpret_cast<uint32_t*>(d) = v;
          if ((n0 >> 6) == other) cluster_store(cluster_addr(d, other), v);
        }
      }
    };
    back(std::integral_constant<int, 2>());
    __syncthreads();
    dense16x16<false>(s->dz[2] + row0 * kRow, s->W3, n0, lane, acc);
    back(std::integral_constant<int, 1>());
    __syncthreads();
    dense16x16<false>(s->dz[1] + row0 * kRow, s->W2, n0, lane, acc);
    back(std::integral_constant<int, 0>());
    cluster_barrier();   // both blocks' operands are complete
    // ---- weight gradients of this block's 64 output units (of layer 4: half the n tiles)
    {
      float* out = part + (size_t)p * kPart;
      float* W2g = out + kEnc * kH;
      float* W3g = W2g + kH * kH;
      float* W4g = W3g + kH * kH;
      float* bg = out + kMlpNW;
      const int w = warp & 3, m0 = half0 + 16 * w;      // its m tile
      // 17 n tiles of each of dW_2 and dW_3, 5 of dW_1, and of dW_4's 17 nine for block 0 (3, 2, 2, 2), eight for block 1
      if (warp < 4) {
        grad_tiles64<9, kH, kH>(s->dz[1], kRow, m0, s->a[0], kRow, 0, lane, W2g, bg + kH);
        if (crank == 0 && w == 0)
          grad_tiles64<3, 3, kH>(s->dy, kRowY, 0, s->a[2], kRow, 0, lane, W4g, bg + 3 * kH);
        else
          grad_tiles64<2, 3, kH>(s->dy, kRowY, 0, s->a[2], kRow, crank == 0 ? 2 * w + 1 : 9 + 2 * w, lane, W4g,
                                 bg + 3 * kH);
      } else if (warp < 8) {
        grad_tiles64<8, kH, kH>(s->dz[1], kRow, m0, s->a[0], kRow, 9, lane, W2g, bg + kH);
        grad_tiles64<2, kH, kEnc>(s->dz[0], kRow, m0, s->a0, kRow0, 0, lane, out, bg);
      } else if (warp < 12) {
        grad_tiles64<9, kH, kH>(s->dz[2], kRow, m0, s->a[1], kRow, 0, lane, W3g, bg + 2 * kH);
        grad_tiles64<1, kH, kEnc>(s->dz[0], kRow, m0, s->a0, kRow0, 4, lane, out, bg);
      } else {
        grad_tiles64<8, kH, kH>(s->dz[2], kRow, m0, s->a[1], kRow, 9, lane, W3g, bg + 2 * kH);
        grad_tiles64<2, kH, kEnc>(s->dz[0], kRow, m0, s->a0, kRow0, 2, lane, out, bg);
      }
    }
    if (p + (int)(gridDim.x >> 1) < parts) cluster_barrier();   // before the operands are written again
  }
}

struct AdamArgs {
  float *W, *b, *adam;
  float lr, beta1, beta2, eps, c1, c2;
  uint16_t *Wbf, *W2t, *W3t;
};

// The parts of the gradient added in order; with ADAM the step on the FP32
// masters (which rewrites the BF16 copies and the transposes of W2 and W3),
// without it into gW, gb.  The last block takes the loss: the rows'
// squared errors in a fixed order.
template <bool ADAM>
__global__ void __launch_bounds__(kStepThreads) k_mlp_step(const float* __restrict__ part, int nparts, int stride, AdamArgs ad,
                                                         float* __restrict__ gW, float* __restrict__ gb,
                                                         const float* __restrict__ err, int B,
                                                         float* __restrict__ loss) {
  constexpr int n_all = (int)(kMlpNW + kMlpNB);
  if ((int)blockIdx.x * kStepThreads >= n_all) {
    __shared__ double sh[kStepThreads];
    double v = 0.0;
    for (int i = threadIdx.x; i < B; i += kStepThreads) v += err[i];
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int o = kStepThreads / 2; o > 0; o >>= 1) {
      if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
      __syncthreads();
    }
    if (threadIdx.x == 0) *loss = (float)(sh[0] / (3.0 * B));
    return;
  }
  const int i = (int)blockIdx.x * kStepThreads + threadIdx.x;
  if (i >= n_all) return;
  float gr = 0.0f;
#pragma unroll 16
  for (int c = 0; c < nparts; ++c) gr += part[(size_t)c * stride + i];
  if (!ADAM) {
    if (i < kMlpNW) gW[i] = gr;
    else gb[i - kMlpNW] = gr;
    return;
  }
  // moments: W's first, W's second, b's first, b's second
  const bool bias = i >= kMlpNW;
  float* m_ = ad.adam + (bias ? kMlpNW + i : i);
  float* v_ = m_ + (bias ? kMlpNB : kMlpNW);
  float* w_ = bias ? ad.b + (i - kMlpNW) : ad.W + i;
  const float m = ad.beta1 * *m_ + (1.0f - ad.beta1) * gr;
  const float v = ad.beta2 * *v_ + (1.0f - ad.beta2) * gr * gr;
  *m_ = m;
  *v_ = v;
  const float w = *w_ - ad.lr * (m / ad.c1) / (sqrtf(v / ad.c2) + ad.eps);
  *w_ = w;
  if (bias) return;
  const uint16_t bits = bf16_bits(w);
  ad.Wbf[i] = bits;
  const int o2 = kEnc * kH, o3 = o2 + kH * kH;
  if (i >= o2 && i < o3) ad.W2t[((i - o2) % kH) * kH + (i - o2) / kH] = bits;
  else if (i >= o3 && i < o3 + kH * kH) ad.W3t[((i - o3) % kH) * kH + (i - o3) / kH] = bits;
}

unsigned step_blocks(const float* loss) {
  return (unsigned)((kMlpNW + kMlpNB + kStepThreads - 1) / kStepThreads) + (loss ? 1u : 0u);
}

}  // namespace

int mlp_grad_parts(int B) { return (int)(((int64_t)B + kTrRows - 1) / kTrRows); }

cudaError_t mlp_train_partials(const MlpArgs& a, const float* x0, const float* xT, int B, float* err, float* part,
                               cudaStream_t st) {
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem))))
    return e;
  int dev = 0, sms = 2;
  if ((e = cudaGetDevice(&dev)) || (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev))) return e;
  const int parts = mlp_grad_parts(B), pairs = sms / 2 > 0 ? sms / 2 : 1;
  k_mlp_train<<<2 * (unsigned)(parts < pairs ? parts : pairs), kTrThreads, sizeof(TrainSmem), st>>>(a, x0, xT, B,
                                                                                                   parts, err, part);
  return cudaGetLastError();
}

cudaError_t mlp_sum_partials(const float* part, int nparts, int stride, float* gW, float* gb, const float* err, int B, float* loss,
                             cudaStream_t st) {
  k_mlp_step<false><<<step_blocks(loss), kStepThreads, 0, st>>>(part, nparts, stride, AdamArgs{}, gW, gb, err, B, loss);
  return cudaGetLastError();
}

cudaError_t mlp_adam_step(const pdmp_mlp* net, const float* part, int nparts, float lr, float beta1, float beta2,
                          float eps, int step, const float* err, int B, float* loss, cudaStream_t st) {
  const AdamArgs ad{net->W, net->b, net->adam, lr, beta1, beta2, eps, 1.0f - powf(beta1, (float)step),
                    1.0f - powf(beta2, (float)step), net->W_bf16, net->Wt_bf16, net->Wt_bf16 + kH * kH};
  k_mlp_step<true><<<step_blocks(loss), kStepThreads, 0, st>>>(part, nparts, kPart, ad, nullptr, nullptr, err, B, loss);
  return cudaGetLastError();
}

}  // namespace pdmp
