// The surrogate network's input encoding, shared by its training (mlp_train.cu,
// mlp.cu) and inference (mlp_tc05.cu) kernels, and what the training kernels share.
//
// u = (x - lo) s - 1 with the network's float32 lo and s (in_scale).  The
// encoding is [u_0..u_2, then for k = 0..5: sin(2^k pi u_j), cos(2^k pi u_j)],
// and sin(2^k pi u) = sin(2 pi tau), tau = 2^(k-1) ((x - lo) s - 1).  The
// product w = (x - lo) s is kept as w_hi + w_lo (an FMA gives the rounding
// error of the product exactly), 2^(k-1) w_hi - rint(2^(k-1) w_hi) is exact,
// and the - 2^(k-1) of the shift is an integer for k >= 1 (a half turn for
// k = 0): the only rounded steps left are the addition of the small w_lo term
// and the angle 2 pi r.  Without this, FP32's rounding of u (about 1e-7) would
// reach the k = 5 features multiplied by 32 pi.
#pragma once

#include <cuda_bf16.h>

#include "kernels.cuh"

namespace pdmp {

struct MlpEncIn {
  float whi[3], wlo[3];
};

__device__ __forceinline__ void mlp_enc_prepare(const float* x, const float* lo, const float* s, MlpEncIn& e) {
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const float d = x[j] - lo[j];
    e.whi[j] = d * s[j];
    e.wlo[j] = fmaf(d, s[j], -e.whi[j]);
  }
}

// feature f (0 .. 38) of the encoding; 0 past the end (padding)
template <bool PRECISE>
__device__ __forceinline__ float mlp_enc_feature(int f, const MlpEncIn& e) {
  if (f >= 39) return 0.0f;
  if (f < 3) return (e.whi[f] - 1.0f) + e.wlo[f];
  const int k = (f - 3) / 6, m = (f - 3) % 6, j = m % 3;
  const float sc = 0.5f * (float)(1 << k);               // 2^(k-1), exact
  const float th_ = e.whi[j] * sc;
  float r = (th_ - rintf(th_)) + e.wlo[j] * sc;
  if (k == 0) r -= 0.5f;
  r -= rintf(r);                                        // [-1/2, 1/2] turn
  const float th = 6.28318530717958648f * r;
  if constexpr (PRECISE) return m < 3 ? sinf(th) : cosf(th);
  return m < 3 ? sin_approx(th) : cos_approx(th);
}

// ---- the training kernels (mlp.cu, mlp_train.cu)
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ uint16_t bf16_bits(float x) {
  const __nv_bfloat16 v = __float2bfloat16_rn(x);
  return *reinterpret_cast<const uint16_t*>(&v);
}

__device__ __forceinline__ void mma16816(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ float silu_f(float z) { return z / (1.0f + __expf(-z)); }
__device__ __forceinline__ float silu_grad_f(float z) {
  const float s = 1.0f / (1.0f + __expf(-z));
  return s * (1.0f + z * (1.0f - s));
}

// Device copy of the network (all pointers device; bf16 as raw uint16).
struct MlpArgs {
  const uint16_t* W1;   // 128 x 39
  const uint16_t* W2;   // 128 x 128  [out][in]
  const uint16_t* W3;   // 128 x 128
  const uint16_t* W4;   // 3 x 128
  const uint16_t* W2t;  // 128 x 128  [in][out] (backward)
  const uint16_t* W3t;  // 128 x 128
  const float *b1, *b2, *b3, *b4;   // one after the other
  float lo[3], in_scale[3], out_scale[3];
};

// One gradient of a batch of B pairs is the sum of mlp_grad_parts(B) parts of 64
// samples, each kMlpNW + kMlpNB numbers (weights then biases), `stride` apart.
constexpr int kMlpTrainPart = 38560;   // the training kernel's stride: whole 128-byte lines
static_assert(kMlpTrainPart >= kMlpNW + kMlpNB, "");
int mlp_grad_parts(int B);
// the parts and the rows' squared errors (mlp_train.cu)
cudaError_t mlp_train_partials(const MlpArgs& a, const float* x0, const float* xT, int B, float* err, float* part,
                               cudaStream_t st);
// their sum into gW, gb; with loss (may be null) the mean squared error
cudaError_t mlp_sum_partials(const float* part, int nparts, int stride, float* gW, float* gb, const float* err, int B, float* loss,
                             cudaStream_t st);
// their sum and the Adam step
cudaError_t mlp_adam_step(const pdmp_mlp* net, const float* part, int nparts, float lr, float beta1, float beta2,
                          float eps, int step, const float* err, int B, float* loss, cudaStream_t st);

}  // namespace pdmp
