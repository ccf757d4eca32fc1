// Occupancy fit (Sec. 3.1) for RBF fields in d = 2, 3 on ordered points and
// centres.  The algorithm is fit.cu's (power iteration, then Nesterov
// iterations, bias as a last unregularised weight); its two sweeps per
// iteration, logits = Phi v and gradient = Phi^T r, are one operation with the
// roles exchanged:
//   out(p) = sum_q weight_q 2^(-g' |p - q|^2),
// targets p and sources q being the labelled points and the centres.
//
// Split.  A launch over the centres has few tiles (128 for M = 4096): 16 warps
// share a tile, and of fewer than 77 tiles a cluster of 2 or 4 blocks, each
// block taking every CS-th run of 32 source groups; the first adds the others'
// sums.
//
// Layout.  Both sets are put in Hilbert order once per call (order.cuh: equal
// chunks of at most 16,384, an order that depends on the points alone), as float4s {p_0 ..,
// weight in .w}, with a bounding box and a strongest-source record for every 32
// sources.  A block owns a tile of consecutive targets; its warps share the
// source groups that are near the tile (the two rules of fast_tile.cuh for s)
// and stage them as packed pairs about the tile's centre, in coordinates scaled
// by sqrt(g'): 2d + 1 packed FP32 operations and one ex2 per pair of targets
// and source.
//
// Launches.  The sweep's epilogue finishes the iteration: after the forward
// sweep the residuals, their sum (the bias's gradient) and their groups'
// records, after the backward sweep the gradient, the Nesterov step, the next
// extrapolated point and its records.  So an iteration is two launches (three
// in the power iteration, whose norm needs all of the gradient).
//
// Every sum runs in a fixed order, so a fit is bit-reproducible.
#include "fast_tile.cuh"
#include "kernels.cuh"
#include "order.cuh"

namespace pdmp {

// one set of points as sources: the table, its groups' boxes ({lo}, {hi}) and
// records ({strongest source, log2 of its |weight|})
struct FitSet {
  float4* tab;
  float4* box;
  float4* rec;
  int64_t n;
  int ngroups;
  int chunk;       // points per order chunk: equal chunks, so that none is left with a few points spread over all
};

struct FitState {
  FitSet X, C;
  const uint8_t* y;     // labels in order
  float *w, *wprev;     // M + 1: iterate (wprev: the power iteration's product); the bias is last
  float* vbias;         // the bias of the point in C.tab's weights
  double* rsum;         // per forward block: sum of r
  double* sq;           // per backward block: sum of squares of its products
  double* bpart;        // per forward block: sum of loss terms
  double* scal;         // [0] lambda, [1] alpha, [2] loss
  int nfwd, nbwd;       // their blocks
  float gl2e;
  double inv_n;
  float l2;
};

// group record of 32 consecutive sources, one per lane (ok: the lane has one)
template <int D>
__device__ __forceinline__ void fit_record(const float4& p, float weight, bool ok, float4* rec, int lane) {
  const float a = ok ? fabsf(weight) : 0.0f;
  const bool odd = __any_sync(0xffffffffu, !(a < INFINITY));
  float m = a;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  const int top = __ffs(__ballot_sync(0xffffffffu, a == m)) - 1;
  const int src = top < 0 ? 0 : top;
  const float x = __shfl_sync(0xffffffffu, p.x, src), y = __shfl_sync(0xffffffffu, p.y, src),
              z = __shfl_sync(0xffffffffu, p.z, src);
  if (lane == 0) *rec = make_float4(x, y, z, odd ? INFINITY : (m > 0.0f ? log2f(m) : -INFINITY));
}

// Clusters [0, xc): chunks of the points; [xc, xc + cc): chunks of the centres.
template <int D>
__global__ void __cluster_dims__(kOrderBlocks, 1, 1) __launch_bounds__(kOrderThreads)
    k_fit_order(const float* __restrict__ X, const uint8_t* __restrict__ y, int xc, const float* __restrict__ centres,
                FitSet xs, FitSet cs, uint8_t* __restrict__ ys, int32_t* __restrict__ cperm, int xbits, int cbits,
                float w0, float* __restrict__ vbias) {
  __shared__ OrderSmem s;
  const int cluster = (int)(blockIdx.x / kOrderBlocks), crank = (int)(blockIdx.x % kOrderBlocks);
  const bool is_x = cluster < xc;
  if (blockIdx.x == 0 && threadIdx.x == 0) *vbias = w0;
  const FitSet f = is_x ? xs : cs;
  const int64_t m0 = (int64_t)(is_x ? cluster : cluster - xc) * f.chunk;
  const float* pts = (is_x ? X : centres) + m0 * D;
  const int n = (int)min64(f.chunk, f.n - m0);
  const int share = cluster_order<D>(pts, n, is_x ? xbits : cbits, s, crank);
  const int lane = threadIdx.x & 31, p0 = crank * share, end = n < p0 + share ? n : p0 + share;
  for (int g = p0 / kGroup + (threadIdx.x >> 5); g * kGroup < end; g += kOrderWarps) {
    const int i = g * kGroup + lane;
    const bool ok = i < end;
    float4 p = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    float lo[D], hi[D];
    bool odd = false;
    if (ok) {
      const int m = (int)(s.items[i - p0] & (kOrderChunk - 1));
      p.x = pts[(size_t)m * D];
      p.y = pts[(size_t)m * D + 1];
      if (D == 3) p.z = pts[(size_t)m * D + D - 1];
      if (is_x) {
        ys[m0 + i] = y[m0 + m];
      } else {
        cperm[m0 + i] = (int32_t)(m0 + m);
        p.w = w0;
      }
      f.tab[m0 + i] = p;
    }
    const float v[3] = {p.x, p.y, p.z};
#pragma unroll
    for (int j = 0; j < D; ++j) {
      lo[j] = ok ? v[j] : INFINITY;
      hi[j] = ok ? v[j] : -INFINITY;
      odd = odd || (ok && !(fabsf(v[j]) < INFINITY));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        lo[j] = fminf(lo[j], __shfl_xor_sync(0xffffffffu, lo[j], o));
        hi[j] = fmaxf(hi[j], __shfl_xor_sync(0xffffffffu, hi[j], o));
      }
    }
    odd = __any_sync(0xffffffffu, odd);
    float4* box = f.box + 2 * (m0 / kGroup + g);
    if (lane == 0) {
      const float big = INFINITY;
      box[0] = odd ? make_float4(-big, -big, -big, 0.0f) : make_float4(lo[0], lo[1], D == 3 ? lo[D - 1] : 0.0f, 0.0f);
      box[1] = odd ? make_float4(big, big, big, 0.0f) : make_float4(hi[0], hi[1], D == 3 ? hi[D - 1] : 0.0f, 0.0f);
    }
    if (!is_x) fit_record<D>(p, w0, ok, f.rec + m0 / kGroup + g, lane);
  }
}

enum FitMode { kFitPower, kFitGradient, kFitLoss };

// Tile shapes: 32 K / SUB targets (K per lane in packed pairs; SUB = 2: the half
// warps hold the same targets and take every other source of a group).
constexpr int kFitAhead = 4;     // groups in flight per warp
constexpr int kFitWarps = 8, kFitCentreWarps = 16;
template <int D, int K, int SUB, int W>
struct FitTile {
  static constexpr int kT = 32 * K / SUB, kRec = 4;   // u64 per staged source
  static constexpr size_t kStage = (size_t)2 * kGroup * kRec * 8, kRaw = (size_t)kFitAhead * kGroup * sizeof(float4);
  static constexpr size_t kSums = (size_t)W * kT * sizeof(float);
  static constexpr size_t kSmem = W * (kStage + kRaw) + kSums + sizeof(NearSmem);
};

// Sums over the near sources of a tile of targets, shared by the CS blocks of a
// cluster (this one of rank crank); in the block of rank 0 thread t < kT returns
// the total of target t (0 past the end).
template <int D, int K, int SUB, int W, int CS>
__device__ __forceinline__ double fit_sweep(const FitSet& tgt, const FitSet& src, float gl2e, unsigned char* smem,
                                            int crank) {
  using F = FitTile<D, K, SUB, W>;
  constexpr int P = K / 2, T = F::kT, half = 32 / SUB;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  u64* stage = reinterpret_cast<u64*>(smem) + (size_t)warp * 2 * kGroup * F::kRec;
  float4* raw = reinterpret_cast<float4*>(smem + W * F::kStage) + (size_t)warp * kFitAhead * kGroup;
  float* sums = reinterpret_cast<float*>(smem + W * (F::kStage + F::kRaw));
  NearSmem& ns = *reinterpret_cast<NearSmem*>(sums + W * T);
  const int64_t t0 = (int64_t)(blockIdx.x / CS) * T;
  // this block's groups, numbered j: runs of 32, every CS-th run of the set
  const int runs = (src.ngroups + 31) / 32, own = (runs - crank + CS - 1) / CS * 32;
  auto group = [&](int j) { return CS == 1 ? j : ((j >> 5) * CS + crank) << 5 | (j & 31); };

  // the lane's targets, the tile's box and its centre
  float x[K][D], lo[D], hi[D], o[D];
  bool odd = false;
#pragma unroll
  for (int j = 0; j < D; ++j) { lo[j] = INFINITY; hi[j] = -INFINITY; }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int64_t i = t0 + k * half + lane % half;
    const float4 p = tgt.tab[i < tgt.n ? i : tgt.n - 1];   // past the end: the last target again
    const float v[3] = {p.x, p.y, p.z};
#pragma unroll
    for (int j = 0; j < D; ++j) {
      x[k][j] = v[j];
      lo[j] = fminf(lo[j], v[j]);
      hi[j] = fmaxf(hi[j], v[j]);
      odd = odd || !(fabsf(v[j]) < INFINITY);
    }
  }
#pragma unroll
  for (int j = 0; j < D; ++j) {
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
      lo[j] = fminf(lo[j], __shfl_xor_sync(0xffffffffu, lo[j], s));
      hi[j] = fmaxf(hi[j], __shfl_xor_sync(0xffffffffu, hi[j], s));
    }
    const float c = 0.5f * (lo[j] + hi[j]);
    o[j] = c - c == 0.0f ? c : 0.0f;
  }
  odd = __any_sync(0xffffffffu, odd);
  const float sc = sqrtf(gl2e);
  u64 U[P][D], S[P];
#pragma unroll
  for (int i = 0; i < P; ++i) {
#pragma unroll
    for (int j = 0; j < D; ++j) U[i][j] = pk(sc * (x[2 * i][j] - o[j]), sc * (x[2 * i + 1][j] - o[j]));
    S[i] = 0ull;
  }

  // near groups: rule (1) at exponent -127, rule (2) for the sum alone
  float ref = -INFINITY;
#pragma unroll 2
  for (int j = warp * 32 + lane; j < own; j += W * 32) {
    const int g = group(j);
    if (g >= src.ngroups) continue;
    const float4 b = src.rec[g];
    const float mu[3] = {b.x, b.y, b.z};
    float d2 = 0.0f;
#pragma unroll
    for (int j = 0; j < D; ++j) {
      const float reach = fmaxf(hi[j] - mu[j], mu[j] - lo[j]);
      d2 = fmaf(reach, reach, d2);
    }
    ref = fmaxf(ref, fmaf(-gl2e, d2, b.w));
  }
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) ref = fmaxf(ref, __shfl_xor_sync(0xffffffffu, ref, s));
  if (lane == 0) ns.refs[warp] = ref;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < W; ++w) ref = fmaxf(ref, ns.refs[w]);
  if (CS > 1) {                  // the cluster's: rank r's in word r of every block
    float* all = ns.state;
    if ((int)threadIdx.x < CS) cluster_store(cluster_addr(&all[crank], (int)threadIdx.x), __float_as_uint(ref));
    cluster_barrier();
#pragma unroll
    for (int r = 0; r < CS; ++r) ref = fmaxf(ref, all[r]);
  }
  const float lim1 = odd ? INFINITY : 127.0f, lim2 = odd ? INFINITY : 30.0f + lg2_approx((float)src.n) - ref;
  auto near = [&](int j) {
    const int g = group(j);
    if (g >= src.ngroups) return false;
    const float4 b0 = src.box[2 * g], b1 = src.box[2 * g + 1];
    const float blo[3] = {b0.x, b0.y, b0.z}, bhi[3] = {b1.x, b1.y, b1.z}, lw = src.rec[g].w;
    float d2 = 0.0f;
#pragma unroll
    for (int j = 0; j < D; ++j) {
      const float gap = fmaxf(0.0f, fmaxf(blo[j] - hi[j], lo[j] - bhi[j]));
      d2 = fmaf(gap, gap, d2);
    }
    const float y = gl2e * d2;
    // rule (1) takes phi alone: a weight of any size times an exact zero is zero unless it is not finite
    // (a group with a point that is not finite has the box of everything, and stays)
    return !((y > lim1 && lw < INFINITY) || y - lw > lim2) || b0.x == -INFINITY;
  };
  // the near sources, kFitAhead groups in flight per warp (a group's sums take
  // less than its load)
  for (int g0 = 0; g0 < own; g0 += kNearBatch) {
    if (g0 > 0) __syncthreads();   // every warp has walked the batch before
    const int n = near_list<W>(ns, g0, own, warp, lane, near);
    const int cnt = warp < n ? (n - warp + W - 1) / W : 0;
    auto prefetch = [&](int j) {   // a lane's entry is its own: read before its slot's next prefetch
      if (j < cnt) {
        const int64_t i = (int64_t)group(g0 + ns.list[warp + j * W]) * kGroup + lane;
        if (i < src.n) cp_async16(raw + (j % kFitAhead) * kGroup + lane, src.tab + i);
      }
      cp_async_commit();
    };
    auto fetch = [&](int j) {      // group j's source of this lane (past the end: weight 0 at the centre)
      asm volatile("cp.async.wait_group %0;" ::"n"(kFitAhead - 1) : "memory");
      const int64_t i = (int64_t)group(g0 + ns.list[warp + j * W]) * kGroup + lane;
      return i < src.n ? raw[(j % kFitAhead) * kGroup + lane] : make_float4(o[0], o[1], o[D - 1], 0.0f);
    };
    auto build = [&](const float4& p, int b) {
      const float v[3] = {p.x, p.y, p.z};
      u64* r = stage + ((size_t)b * kGroup + lane) * F::kRec;
      u64 q[4];
#pragma unroll
      for (int j = 0; j < D; ++j) {
        const float c = -sc * (v[j] - o[j]);
        q[j] = pk(c, c);
      }
      q[D] = pk(p.w, p.w);
      if (D == 2) q[3] = 0ull;
      *reinterpret_cast<ulonglong2*>(r) = make_ulonglong2(q[0], q[1]);
      *reinterpret_cast<ulonglong2*>(r + 2) = make_ulonglong2(q[2], q[3]);
    };
#pragma unroll
    for (int j = 0; j < kFitAhead; ++j) prefetch(j);
    if (cnt > 0) build(fetch(0), 0);
    prefetch(kFitAhead);
    __syncwarp();
    for (int j = 0; j < cnt; ++j) {
      float4 p = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (j + 1 < cnt) p = fetch(j + 1);
      prefetch(j + 1 + kFitAhead);
      const u64* rec = stage + (size_t)(j & 1) * kGroup * F::kRec + (SUB == 2 && lane >= half ? F::kRec : 0);
#pragma unroll 8
      for (int c = 0; c < kGroup / SUB; ++c) {
        const ulonglong2 a0 = *reinterpret_cast<const ulonglong2*>(rec + (size_t)c * SUB * F::kRec);
        const ulonglong2 a1 = *reinterpret_cast<const ulonglong2*>(rec + (size_t)c * SUB * F::kRec + 2);
        const u64 r[4] = {a0.x, a0.y, a1.x, a1.y};
#pragma unroll
        for (int i = 0; i < P; ++i) {
          u64 dx = add2(U[i][0], r[0]);
          u64 q = mul2(dx, dx);
#pragma unroll
          for (int j2 = 1; j2 < D; ++j2) {
            dx = add2(U[i][j2], r[j2]);
            q = fma2(dx, dx, q);
          }
          S[i] = fma2(r[D], ex2x2_neg(q), S[i]);
        }
      }
      if (j + 1 < cnt) build(p, (j + 1) & 1);
      __syncwarp();
    }
    cp_async_wait_all();
  }
#pragma unroll
  for (int i = 0; i < P; ++i) {
    float v[2];
    upk(S[i], v[0], v[1]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (SUB == 2) v[h] += __shfl_xor_sync(0xffffffffu, v[h], 16);
      if (lane < half) sums[warp * T + (2 * i + h) * half + lane] = v[h];
    }
  }
  __syncthreads();
  double acc = 0.0;
  if ((int)threadIdx.x < T && t0 + threadIdx.x < tgt.n)
#pragma unroll
    for (int w = 0; w < W; ++w) acc += (double)sums[w * T + threadIdx.x];
  if (CS > 1) {
    double* part = reinterpret_cast<double*>(smem);      // [CS][T] in rank 0, over its stages (read)
    cluster_barrier();                                   // rank 0 has read its stages
    if (crank > 0 && (int)threadIdx.x < T) {
      const uint32_t at = cluster_addr(&part[crank * T + threadIdx.x], 0);
      const unsigned long long v = (unsigned long long)__double_as_longlong(acc);
      cluster_store(at, (uint32_t)v);
      cluster_store(at + 4, (uint32_t)(v >> 32));
    }
    cluster_barrier();
    if (crank == 0 && (int)threadIdx.x < T)
#pragma unroll
      for (int r = 1; r < CS; ++r) acc += part[r * T + threadIdx.x];
  }
  return acc;
}

// sum of one double per thread over the block, in a fixed order (sh: 32 doubles); every thread returns it
__device__ __forceinline__ double block_sum(double v, double* sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  double t = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0.0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  __syncthreads();
  return t;
}

// logits of a tile of points, then (power iteration) r = logit or r = sigmoid(logit) - y, or the loss terms
template <int D, int K, int MODE>
__global__ void __launch_bounds__(32 * kFitWarps, 2) k_fit_points(FitState f) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double sh[32];
  constexpr int T = FitTile<D, K, 1, kFitWarps>::kT;
  const double acc = fit_sweep<D, K, 1, kFitWarps, 1>(f.X, f.C, f.gl2e, smem, 0);
  const int lane = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * T + threadIdx.x;
  const bool ok = (int)threadIdx.x < T && i < f.X.n;
  float r = 0.0f;
  double term = 0.0;
  if (ok) {
    const float l = (float)acc + f.vbias[0];
    if (MODE == kFitPower) {
      r = l;
    } else {
      const float yi = f.y[i] ? 1.0f : 0.0f;
      r = sigmoid_f(l) - yi;
      if (MODE == kFitLoss) {
        const double ld = (double)l;
        term = (ld > 0 ? ld + log1p(exp(-ld)) : log1p(exp(ld))) - (double)yi * ld;
      }
    }
  }
  if (MODE == kFitLoss) {
    const double t = block_sum(term, sh);
    if (threadIdx.x == 0) f.bpart[blockIdx.x] = t;
    return;
  }
  if ((int)threadIdx.x < T) {
    float4 p = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (ok) {
      p = f.X.tab[i];
      f.X.tab[i].w = r;
    }
    const int64_t g = i / kGroup;
    if (g < f.X.ngroups) fit_record<D>(p, r, ok, f.X.rec + g, lane);
  }
  const double t = block_sum((double)r, sh);
  if (threadIdx.x == 0) f.rsum[blockIdx.x] = t;
}

// gradient of a tile of centres, then the power iteration's product or the
// Nesterov step k (1-based) and the point the next forward sweep is taken at
template <int D, int CS, int MODE>
__global__ void __launch_bounds__(32 * kFitCentreWarps, 1) k_fit_centres(FitState f, int k, int last) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double sh[32];
  constexpr int T = FitTile<D, 2, 2, kFitCentreWarps>::kT;
  const int tile = (int)(blockIdx.x / CS), crank = (int)(blockIdx.x % CS);
  const double acc = fit_sweep<D, 2, 2, kFitCentreWarps, CS>(f.C, f.X, f.gl2e, smem, crank);
  if (crank > 0) return;         // nobody reads this block any more
  const int lane = threadIdx.x & 31;
  const int64_t M = f.C.n, m = (int64_t)tile * T + threadIdx.x;
  const bool ok = (int)threadIdx.x < T && m < M;
  // v = w + beta (w - wprev) with beta = (k - 1) / (k + 2) for step k: the next step's
  const float beta = last ? 0.0f : (float)k / (float)(k + 3);
  double sq = 0.0;
  if ((int)threadIdx.x < T) {
    float4 p = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    float v = 0.0f;
    if (ok) {
      p = f.C.tab[m];
      const float g = (float)(acc * f.inv_n);
      if (MODE == kFitPower) {
        f.wprev[m] = g;
        sq = (double)g * (double)g;
      } else {
        const float wn = fmaf(-(float)f.scal[1], fmaf(f.l2, p.w, g), p.w), wo = f.w[m];
        v = fmaf(beta, wn - wo, wn);
        f.w[m] = wn;
        f.C.tab[m].w = v;
      }
    }
    const int64_t g = m / kGroup;
    if (MODE != kFitPower && g < f.C.ngroups) fit_record<D>(p, v, ok, f.C.rec + g, lane);
  }
  if (MODE == kFitPower) {
    const double t = block_sum(sq, sh);
    if (threadIdx.x == 0) f.sq[tile] = t;
  }
  if (blockIdx.x == 0) {       // the bias: its feature is 1
    double s = 0.0;
    for (int b = threadIdx.x; b < f.nfwd; b += blockDim.x) s += f.rsum[b];
    s = block_sum(s, sh);
    if (threadIdx.x == 0) {
      const float g = (float)(s * f.inv_n);
      if (MODE == kFitPower) {
        f.wprev[M] = g;
      } else {
        const float wn = fmaf(-(float)f.scal[1], g, f.vbias[0]), wo = f.w[M];
        f.w[M] = wn;
        f.vbias[0] = fmaf(beta, wn - wo, wn);
      }
    }
  }
}

// v = product / |product|, lambda = |product|, alpha = 1 / (lambda / 4 + l2); after the last power iteration
// (last) the weights start at zero instead
template <int D>
__global__ void __launch_bounds__(256) k_fit_unit(FitState f, int last) {
  __shared__ double sh[32];
  const int64_t M = f.C.n;
  double s = 0.0;
  for (int b = threadIdx.x; b < f.nbwd; b += blockDim.x) s += f.sq[b];
  s = block_sum(s, sh) + (double)f.wprev[M] * (double)f.wprev[M];
  const double nrm = sqrt(s);
  const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, g = m / kGroup;
  const bool ok = m < M;
  float4 p = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  float v = 0.0f;
  if (ok) {
    p = f.C.tab[m];
    v = last ? 0.0f : (nrm > 0.0 ? (float)((double)f.wprev[m] / nrm) : p.w);
    f.C.tab[m].w = v;
    if (last) f.w[m] = 0.0f;
  }
  if (g < f.C.ngroups) fit_record<D>(p, v, ok, f.C.rec + g, threadIdx.x & 31);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (last) {
      f.w[M] = 0.0f;
      f.vbias[0] = 0.0f;
    } else if (nrm > 0.0) {
      f.vbias[0] = (float)((double)f.wprev[M] / nrm);
    }
    f.scal[0] = nrm;
    f.scal[1] = 1.0 / (0.25 * nrm + (double)f.l2);
  }
}

// one block: scal[2] = loss + (l2 / 2) |w|^2
__global__ void __launch_bounds__(1024) k_fit_total(FitState f) {
  __shared__ double sh[32];
  double a = 0.0, b = 0.0;
  for (int q = threadIdx.x; q < f.nfwd; q += blockDim.x) a += f.bpart[q];
  for (int64_t m = threadIdx.x; m < f.C.n; m += blockDim.x) b += (double)f.w[m] * (double)f.w[m];
  a = block_sum(a, sh);
  b = block_sum(b, sh);
  if (threadIdx.x == 0) {
    const double loss = a * f.inv_n + 0.5 * (double)f.l2 * b;
    f.scal[2] = loss;
    if (!isfinite(loss)) raise_flag(FLAG_FIT_NONFINITE);
  }
}

__global__ void k_fit_unorder(const float* __restrict__ w, const int32_t* __restrict__ perm, int64_t M,
                              float* __restrict__ out) {
  const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (m < M) out[perm[m]] = w[m];
}

// ------------------------------------------------------------------ host
// Points: 128-sample tiles once they fill the GPU, else 64.  Centres: tiles of
// 32.  Measured (2-D, n = 50,000, M = 4096, a third of the pairs near): 25 us a
// launch over the points, 33 us over the centres, 8 us of each the launch and
// the tile's set-up; all pairs near (points within one feature width) 54 and 70
// us, 0.4 of the ex2 rate.  Clusters over all sizes (42 us), tiles dealt out
// across the domain (25 and 41) and launches overlapped by programmatic
// dependence (a fifth slower) brought nothing.
static bool fit_wide_points(int64_t n) { return n >= 128 * 304; }

static size_t al256(size_t b) { return (b + 255) & ~size_t(255); }

size_t fit_rbf_workspace(int64_t M, int64_t n) {
  const size_t gx = (size_t)group_count(n), gc = (size_t)group_count(M);
  return al256(sizeof(float4) * (size_t)n) + al256(sizeof(float4) * 2 * gx) + al256(sizeof(float4) * gx) +
         al256(sizeof(float4) * (size_t)M) + al256(sizeof(float4) * 2 * gc) + al256(sizeof(float4) * gc) +
         al256((size_t)n) + al256(sizeof(int32_t) * (size_t)M) + 2 * al256(sizeof(float) * (size_t)(M + 1)) +
         al256(sizeof(float)) + 2 * al256(sizeof(double) * (size_t)((n + 63) / 64)) +
         al256(sizeof(double) * (size_t)((M + 31) / 32)) + al256(sizeof(double) * 8);
}

template <typename Fn, typename... A>
static cudaError_t launch_tiles(Fn fn, int64_t tiles, int cs, int warps, size_t smem, cudaStream_t st, A... args) {
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3((unsigned)(tiles * cs));
  c.blockDim = dim3(32u * (unsigned)warps);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cs;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  c.attrs = at;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, fn, args...);
}

template <int D, int MODE>
static cudaError_t launch_points(const FitState& f, cudaStream_t st) {
  if (fit_wide_points(f.X.n))
    return launch_tiles(k_fit_points<D, 4, MODE>, f.nfwd, 1, kFitWarps, FitTile<D, 4, 1, kFitWarps>::kSmem, st, f);
  return launch_tiles(k_fit_points<D, 2, MODE>, f.nfwd, 1, kFitWarps, FitTile<D, 2, 1, kFitWarps>::kSmem, st, f);
}

template <int D, int MODE>
static cudaError_t launch_centres(const FitState& f, int k, bool last, cudaStream_t st) {
  constexpr size_t smem = FitTile<D, 2, 2, kFitCentreWarps>::kSmem;
  constexpr int W = kFitCentreWarps;
  const int l = last ? 1 : 0;
  if (f.nbwd <= 38) return launch_tiles(k_fit_centres<D, 4, MODE>, f.nbwd, 4, W, smem, st, f, k, l);
  if (f.nbwd <= 76) return launch_tiles(k_fit_centres<D, 2, MODE>, f.nbwd, 2, W, smem, st, f, k, l);
  return launch_tiles(k_fit_centres<D, 1, MODE>, f.nbwd, 1, W, smem, st, f, k, l);
}

template <int D>
static cudaError_t fit_run(const FieldArgs& geom, const float* X, const uint8_t* y, int64_t n, float l2,
                           int power_iters, int iters, float* w_out, float* bias_out, float* loss_out,
                           float* alpha_out, void* ws, cudaStream_t st) {
  const int64_t M = geom.M;
  char* p = (char*)ws;
  auto take = [&](size_t b) { char* q = p; p += al256(b); return q; };
  FitState f{};
  f.X.n = n;
  f.X.ngroups = group_count(n);
  f.C.n = M;
  f.C.ngroups = group_count(M);
  for (FitSet* s : {&f.X, &f.C}) {
    s->tab = (float4*)take(sizeof(float4) * (size_t)s->n);
    s->box = (float4*)take(sizeof(float4) * 2 * (size_t)s->ngroups);
    s->rec = (float4*)take(sizeof(float4) * (size_t)s->ngroups);
  }
  uint8_t* ys = (uint8_t*)take((size_t)n);
  int32_t* cperm = (int32_t*)take(sizeof(int32_t) * (size_t)M);
  f.y = ys;
  f.w = (float*)take(sizeof(float) * (size_t)(M + 1));
  f.wprev = (float*)take(sizeof(float) * (size_t)(M + 1));
  f.vbias = (float*)take(sizeof(float));
  f.rsum = (double*)take(sizeof(double) * (size_t)((n + 63) / 64));
  f.bpart = (double*)take(sizeof(double) * (size_t)((n + 63) / 64));
  f.sq = (double*)take(sizeof(double) * (size_t)((M + 31) / 32));
  f.scal = (double*)take(sizeof(double) * 8);
  const int tx = fit_wide_points(n) ? 128 : 64, tc = 32;
  f.nfwd = (int)((n + tx - 1) / tx);
  f.nbwd = (int)((M + tc - 1) / tc);
  f.gl2e = geom.gamma * kLog2e;
  f.inv_n = 1.0 / (double)n;
  f.l2 = l2;

  auto chunks = [](FitSet& s) {   // whole groups, and whole tiles, per chunk
    const int64_t c = (s.n + kOrderChunk - 1) / kOrderChunk, each = ((s.n + c - 1) / c + 127) / 128 * 128;
    s.chunk = (int)each;
    return (int)((s.n + each - 1) / each);
  };
  const int xc = chunks(f.X), cc = chunks(f.C);
  const float w0 = (float)(1.0 / sqrt((double)(M + 1)));
  k_fit_order<D><<<(unsigned)(xc + cc) * kOrderBlocks, kOrderThreads, 0, st>>>(
      X, y, xc, geom.centres, f.X, f.C, ys, cperm, sort_bits(D, n < f.X.chunk ? n : f.X.chunk),
      sort_bits(D, M < f.C.chunk ? M : f.C.chunk), w0, f.vbias);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;

  for (int it = 0; it < power_iters; ++it) {
    if ((e = launch_points<D, kFitPower>(f, st)) != cudaSuccess) return e;
    if ((e = launch_centres<D, kFitPower>(f, 0, false, st)) != cudaSuccess) return e;
    k_fit_unit<D><<<(unsigned)((M + 255) / 256), 256, 0, st>>>(f, it + 1 == power_iters ? 1 : 0);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  for (int k = 1; k <= iters; ++k) {
    if ((e = launch_points<D, kFitGradient>(f, st)) != cudaSuccess) return e;
    if ((e = launch_centres<D, kFitGradient>(f, k, k == iters, st)) != cudaSuccess) return e;
  }
  if ((e = launch_points<D, kFitLoss>(f, st)) != cudaSuccess) return e;
  k_fit_total<<<1, 1024, 0, st>>>(f);
  k_fit_unorder<<<(unsigned)((M + 255) / 256), 256, 0, st>>>(f.w, cperm, M, w_out);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (bias_out || loss_out || alpha_out) {
    float b;
    double sc[3];
    if ((e = cudaMemcpyAsync(&b, f.w + M, sizeof(float), cudaMemcpyDeviceToHost, st)) != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(sc, f.scal, sizeof(sc), cudaMemcpyDeviceToHost, st)) != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
    if (bias_out) *bias_out = b;
    if (loss_out) *loss_out = (float)sc[2];
    if (alpha_out) *alpha_out = (float)sc[1];
  }
  return cudaSuccess;
}

cudaError_t fit_rbf(int d, const FieldArgs& geom, const float* X, const uint8_t* y, int64_t n, float l2,
                    int power_iters, int iters, float* w_out, float* bias_out, float* loss_out, float* alpha_out,
                    void* ws, cudaStream_t st) {
  if (d == 2)
    return fit_run<2>(geom, X, y, n, l2, power_iters, iters, w_out, bias_out, loss_out, alpha_out, ws, st);
  return fit_run<3>(geom, X, y, n, l2, power_iters, iters, w_out, bias_out, loss_out, alpha_out, ws, st);
}

}  // namespace pdmp
