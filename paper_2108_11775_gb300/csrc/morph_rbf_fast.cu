// Fast RBF morph for d = 2 and d = 3: T Euler steps of Eq. (1) on spatially
// sorted sample tiles.
//
// Expanded exponent.  For a tile with origin o (the centre of its current
// bounding box), u = x - o and c_m = mu_m - o:
//   log2(|w_m| phi_m(x)) = lw_m - g' |u - c_m|^2
//                        = (lw_m - g' |c_m|^2) + 2 g' c_m . u  -  g' |u|^2,
// with g' = gamma log2(e) and lw_m = log2|w_m|.  The last term is the same for
// every feature, so with e'_m = 2^(a_m + b_m . u), a_m = lw_m - g'|c_m|^2 and
// b_m = 2 g' c_m (per tile and step, staged in shared memory):
//   s - bias              = f S,              S = sum_m sg_m e'_m,   f = 2^(-g'|u|^2)
//   sum_m w_m phi_m (x - mu_m) = f (u S - G),  G = sum_m sg_m e'_m c_m
// and grad s = -2 gamma f (u S - G).  A feature then costs 2d + 1 FP32
// operations and one ex2; they run as packed f32x2 instructions over pairs of
// samples.  The rounding error grows with g'|u|^2, so a tile uses the expanded
// form only while g' R^2 <= 8 (R the tile's half-diagonal; about 1.4e-6
// relative error per feature there) and otherwise the direct form x - mu_m
// for that step.
//
// Work split.  A block of 4 warps owns a tile of 320 samples; every warp holds
// all 320 (10 per lane, five f32x2 pairs) and sums over its own contiguous
// quarter of the centres; the four partial sums are added in a fixed order
// once per step.  Launches too small to fill the GPU take 128-sample tiles
// (below).  A sweep visits only the groups of centres that are not exactly
// zero on the tile (fast_tile.cuh, rbf_order.cu).
#include "fast_tile.cuh"
#include "kernels.cuh"
#include "sort.cuh"

namespace pdmp {

template <int D, bool TRACE, int K, int CS>
__global__ void __launch_bounds__(Shape<4, K>::kThreads, Shape<4, K>::kMinBlocks)
k_morph_rbf_fast(TileArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int64_t p0 = (int64_t)(blockIdx.x / CS) * Shape<4, K>::kTile;
  fast_tile<D, 4, K, TRACE, false, CS>(a, p0, a.N, smem, (int)(blockIdx.x % CS));
}

// Samples per lane.  A launch of fewer 320-sample tiles than fit on the GPU at
// once (3 per SM) leaves SMs idle; it takes 128-sample tiles instead (16
// warps per SM).  Measured on a 3-D field (M = 8192, T = 40): 2^16 samples
// 9.3 ms against 13.2 ms; from one wave of 320-sample tiles up the larger tiles
// are as fast or faster in 2-D.  In 3-D a tile's box shrinks slower with the number
// of samples, and small boxes have fewer near groups, so small tiles are kept for
// two thirds more samples (200,000 samples in boxes of 5^3 / 10^3, gamma = 8, M =
// 4096, T = 10: 2.11 / 1.46 ms against 2.21 / 2.04; 400,000: 3.60 / 2.04 against
// 3.52 / 2.86; 2^20: 8.28 / 4.46 against 7.40 / 4.12).
constexpr int kSmallK = 4;

static int num_sms() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                 cudaSuccess || sms < 1)
    sms = 152;
  return sms;
}

// ------------------------------------------------------------------ host
size_t morph_rbf_fast_workspace(int d, int64_t M, int64_t N) { return rbf_order_workspace(d, M, N); }

template <int D, bool TRACE, int K, int CS>
static cudaError_t launch_shape(const TileArgs& a, int64_t N, cudaStream_t st) {
  constexpr size_t smem = tile_smem_bytes<D, 4, K, CS>();
  const unsigned blocks = (unsigned)((N + Shape<4, K>::kTile - 1) / Shape<4, K>::kTile) * CS;
  auto fn = k_morph_rbf_fast<D, TRACE, K, CS>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  if (CS == 1) {
    fn<<<blocks, Shape<4, K>::kThreads, smem, st>>>(a);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(blocks);
  c.blockDim = dim3(Shape<4, K>::kThreads);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CS;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  c.attrs = at;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, fn, a);
}

// 128-sample tiles go to a cluster of 4 blocks while there are fewer tiles than
// SMs, to 2 while there are fewer than two per SM: one block of four warps an
// SM leaves each scheduler a single warp.  Measured (2-D, T = 10): 4096 samples
// and 1024 centres 62 us on clusters of 4; the call with its order 73 us
// against 131 us of one block a tile and the eight-launch sort.
template <int D, bool TRACE>
static cudaError_t launch_tiles(const TileArgs& a, int64_t N, cudaStream_t st) {
  const int64_t sms = num_sms();
  const int64_t tiles = (N + FastShape::kTile - 1) / FastShape::kTile;
  if (tiles >= (D == 3 ? 5 : FastShape::kMinBlocks) * sms) return launch_shape<D, TRACE, FastShape::kK, 1>(a, N, st);
  const int64_t small = (N + Shape<4, kSmallK>::kTile - 1) / Shape<4, kSmallK>::kTile;
  if (small <= sms) return launch_shape<D, TRACE, kSmallK, 4>(a, N, st);
  if (small <= 2 * sms) return launch_shape<D, TRACE, kSmallK, 2>(a, N, st);
  return launch_shape<D, TRACE, kSmallK, 1>(a, N, st);
}

template <int D>
static cudaError_t launch_fast(const FieldArgs& fa, const float* x0, int64_t N, int T, float eta, float* xT,
                               float* ckpt, int k, float* traj, float* steps, void* ws, cudaStream_t st,
                               float* s_out, float* g_out = nullptr) {
  RbfOrder ord;
  cudaError_t e = rbf_order(D, fa.centres, fa.w, fa.M, x0, N, ws, &ord, st);
  if (e != cudaSuccess) return e;
  if (morph_rbf_tc05_eligible(D, N))
    return morph_rbf_tc05(D, fa, x0, ord.perm, N, T, eta, xT, ckpt, k, traj, steps, s_out, g_out, st);
  TileArgs a{};
  a.tab = ord.tab;
  a.box = ord.box;
  a.ngroups = ord.ngroups;
  a.M = fa.M;
  a.gamma = fa.gamma;
  a.bias = fa.bias;
  a.eta = eta;
  a.T = T;
  a.x0 = x0;
  a.perm = ord.perm;
  a.perm_base = 0;
  a.N = N;
  a.xT = xT;
  a.ckpt = ckpt;
  a.kck = k;
  a.traj = traj;
  a.steps = steps;
  a.s_out = s_out;
  a.g_out = g_out;
  return traj != nullptr ? launch_tiles<D, true>(a, N, st) : launch_tiles<D, false>(a, N, st);
}

cudaError_t morph_rbf_fast(int d, const FieldArgs& fa, const float* x0, int64_t N, int T, float eta, float* xT,
                           float* ckpt, int k, float* traj, float* steps, void* ws, cudaStream_t st, float* s_out) {
  if (d == 2) return launch_fast<2>(fa, x0, N, T, eta, xT, ckpt, k, traj, steps, ws, st, s_out);
  if (d == 3) return launch_fast<3>(fa, x0, N, T, eta, xT, ckpt, k, traj, steps, ws, st, s_out);
  return cudaErrorInvalidValue;
}

__global__ void k_query_c(const float* __restrict__ s, int64_t N, float* __restrict__ c) {
  const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (n < N) c[n] = sigmoid_f(s[n]);
}

// s needs N floats of its own when the caller wants c alone
size_t query_rbf_fast_workspace(int d, int64_t M, int64_t N) {
  return morph_rbf_fast_workspace(d, M, N) + ((sizeof(float) * (size_t)N + 255) & ~size_t(255));
}

cudaError_t query_rbf_fast(int d, const FieldArgs& fa, const float* x, int64_t N, float* c, float* s, float* grad,
                           void* ws, cudaStream_t st) {
  if (c != nullptr && s == nullptr) s = (float*)((char*)ws + morph_rbf_fast_workspace(d, fa.M, N));
  // one step with the update discarded, as grad_rbf_fast
  cudaError_t e = d == 2 ? launch_fast<2>(fa, x, N, 1, 0.0f, nullptr, nullptr, 0, nullptr, nullptr, ws, st, s, grad)
                         : launch_fast<3>(fa, x, N, 1, 0.0f, nullptr, nullptr, 0, nullptr, nullptr, ws, st, s, grad);
  if (e != cudaSuccess || c == nullptr) return e;
  k_query_c<<<(unsigned)((N + 255) / 256), 256, 0, st>>>(s, N, c);
  return cudaGetLastError();
}

cudaError_t grad_rbf_fast(int d, const FieldArgs& fa, const float* x, int64_t N, float* g, void* ws,
                          cudaStream_t st) {
  // one step with the update discarded: the per-sample gradient output only
  if (d == 2) return launch_fast<2>(fa, x, N, 1, 0.0f, nullptr, nullptr, 0, nullptr, nullptr, ws, st, nullptr, g);
  if (d == 3) return launch_fast<3>(fa, x, N, 1, 0.0f, nullptr, nullptr, 0, nullptr, nullptr, ws, st, nullptr, g);
  return cudaErrorInvalidValue;
}

}  // namespace pdmp
