// VJP of the T-step map (g_t = (I - eta Hess c(x_t)) g_{t+1}) for RBF fields
// in d = 2, 3 on the forward's spatially sorted tiles.
//
// Segment by segment (last first), the tile's states are recomputed from the
// checkpoint with the forward's tile step and kept in shared memory; each
// step back is one pass over the features at x_t with v = g.  With the
// tile's origin o, u = x - o, c_m = mu_m - o and e'_m = sg_m 2^(a_m + b_m . u)
// (w_m phi_m = f e'_m, f = 2^(-g' |u|^2)), the pass sums the moments
//   S = sum e',  G = sum e' c,  H = sum e' c c^T,
// which give grad s = -2 gamma f (u S - G) and
//   (Hess s) v = 4 gamma^2 f ((u . v)(u S - G) - (u (v . G) - H v)) - 2 gamma f S v
// (sum e' (c . v) = v . G and sum e' (c . v) c = H v, so v enters only per
// sample): 2d + 1 + d(d + 1)/2 packed FP32 operations and one ex2 per sample
// pair and feature, 8 for d = 2.  Tiles too wide for the expanded form take
// the direct form.
//
// Weight gradient (optional).  Sample n adds to d/dw_m, with g = g_{t+1},
//   cA phi_m + cB grad phi_m . g = phi_m (alpha + beta . c_m),
//   cA = -eta sigma'' (grad s . g),  cB = -eta sigma',
//   alpha = cA - 2 gamma cB (u . g),  beta = 2 gamma cB g
// (grad phi_m = -2 gamma phi_m (u - c_m)).  After each Hessian-vector pass
// warp 0 writes u, f alpha and f beta of the tile's samples to shared memory;
// then the sweep is transposed: each lane owns features and sums over the
// tile's sample pairs (phi_m / f = 2^(b_m . u - g' |c_m|^2), 2d + 1 packed
// FP32 operations and one ex2 per pair, as in the forward), so no feature
// needs a reduction across lanes or warps; the block's sums go to its own
// row of the workspace, summed over blocks in a fixed order.
#include "fast_tile.cuh"
#include "kernels.cuh"
#include "sort.cuh"

namespace pdmp {

template <int D>
struct VjRbf {
  static constexpr int kH = D * (D + 1) / 2;           // lower-triangle entries of H
  static constexpr int kUsed = 2 * D + 2 + kH;         // u64 pairs: a, b, sg, c~ = sg c, h = sg c_a c_b
  // whole 16-byte chunks, an odd number of them: the lanes of a quarter warp
  // building consecutive records then write to distinct banks
  static constexpr int kChunks = (kUsed + 1) / 2 % 2 == 1 ? (kUsed + 1) / 2 : (kUsed + 1) / 2 + 1;
  static constexpr int kPairs = 2 * kChunks;
  static constexpr int kSums = 1 + D + kH;             // S, G, H (direct: S, G, P in the first D of H)
  static constexpr int kK = D == 2 ? 8 : 6;
  static constexpr int kW = 4;
  static constexpr int kTile = 32 * kK;
};

template <int D>
__host__ __device__ constexpr size_t vj_rbf_region0() {
  constexpr size_t bufs = (size_t)VjRbf<D>::kW * 2 * kWarpStage * VjRbf<D>::kPairs * 8;
  constexpr size_t red = (size_t)VjRbf<D>::kW * VjRbf<D>::kSums * VjRbf<D>::kTile * 4;
  return bufs > red ? bufs : red;
}
// region 0 (stages / reduction), the raw table entries, the segment's states,
// and with the weight gradient the tile's sample terms (u, f alpha, f beta)
// (and with the cache, the forward's S and G at each of the segment's states)
template <int D>
__host__ __device__ constexpr size_t vj_rbf_smem(int kseg, bool want_gw = false, bool cache = false) {
  return vj_rbf_region0<D>() + (size_t)VjRbf<D>::kW * kWarpStage * FastRec<D>::kTab * sizeof(float4) +
         (size_t)kseg * VjRbf<D>::kTile * D * sizeof(float) +
         (cache ? (size_t)kseg * (1 + D) * VjRbf<D>::kTile * sizeof(float) : 0) +
         (want_gw ? (size_t)(2 * D + 2) * VjRbf<D>::kTile * sizeof(float) : 0);
}

constexpr int kGwFeatures = 4;   // features per lane in the weight-gradient sweep

// Sample terms of the weight-gradient sweep, per pair of samples (2p, 2p + 1):
// 2D + 2 packed pairs [u_0 .. u_{D-1}, f alpha, f beta_0 .. f beta_{D-1}, 0],
// so that a pair's terms are D + 1 16-byte loads.
template <int D>
struct GwTerms {
  static constexpr int kPairs = 2 * D + 2;
  __device__ static void put(float* sm, int s, int slot, float v) {
    sm[((s >> 1) * kPairs + slot) * 2 + (s & 1)] = v;
  }
};

// The weight-gradient sweep of one warp over its near groups of features (sm:
// the tile's sample terms), a feature a lane and kGwFeatures groups at a time;
// adds each feature's sum to row (in table order).
template <int D, int kTile>
__device__ __forceinline__ void vj_gw_sweep(const float4* __restrict__ tab, int64_t M, int g0, NearWalk walk,
                                            bool expanded, const float* o, float gl2e, const float* sm,
                                            float* __restrict__ row, int lane) {
  constexpr int TP = GwTerms<D>::kPairs;
  constexpr int KT = FastRec<D>::kTab;
  constexpr int F = kGwFeatures;
  for (;;) {
    int64_t mf[F];
#pragma unroll
    for (int f = 0; f < F; ++f) {
      const int g = walk.next();
      mf[f] = g < 0 ? M : (int64_t)(g0 + g) * kGroup + lane;
    }
    if (mf[0] >= M && __all_sync(0xffffffffu, mf[0] >= M)) break;
    u64 cst[F], bm[F][D], A[F], Q[F][D];
    float c[F][D];
    bool ok[F];
#pragma unroll
    for (int f = 0; f < F; ++f) {
      const int64_t m = mf[f];
      ok[f] = m < M;
      float mu[D];
      if (ok[f]) {
        const float4 t0 = tab[KT * m];
        mu[0] = t0.x;
        mu[1] = t0.y;
        if (D == 3) mu[2] = t0.z;
      } else {
#pragma unroll
        for (int j = 0; j < D; ++j) mu[j] = o[j];
      }
      float c2 = 0.0f;
#pragma unroll
      for (int j = 0; j < D; ++j) {
        c[f][j] = mu[j] - o[j];   // direct form: o = 0
        c2 = fmaf(c[f][j], c[f][j], c2);
      }
      if (expanded) {   // log2(phi / f) = -g' |c|^2 + 2 g' c . u
        const float a0 = ok[f] ? -gl2e * c2 : -INFINITY;
        cst[f] = pk(a0, a0);
#pragma unroll
        for (int j = 0; j < D; ++j) bm[f][j] = pk(2.0f * gl2e * c[f][j], 2.0f * gl2e * c[f][j]);
      } else {          // log2 phi = -g' |x - mu|^2
        const float nm = ok[f] ? -gl2e : -INFINITY;
        cst[f] = pk(nm, nm);
#pragma unroll
        for (int j = 0; j < D; ++j) bm[f][j] = pk(-mu[j], -mu[j]);
      }
      A[f] = 0ull;
#pragma unroll
      for (int j = 0; j < D; ++j) Q[f][j] = 0ull;
    }
#pragma unroll 2
    for (int p = 0; p < kTile / 2; ++p) {
      const ulonglong2* q = reinterpret_cast<const ulonglong2*>(sm + (size_t)p * TP * 2);
      u64 t[TP];
#pragma unroll
      for (int h = 0; h < TP / 2; ++h) {
        const ulonglong2 v = q[h];
        t[2 * h] = v.x;
        t[2 * h + 1] = v.y;
      }
      u64 up[D], bp[D];
#pragma unroll
      for (int j = 0; j < D; ++j) {
        up[j] = t[j];
        bp[j] = t[D + 1 + j];
      }
      const u64 al = t[D];
#pragma unroll
      for (int f = 0; f < F; ++f) {
        u64 e;
        if (expanded) {
          e = fma2(bm[f][0], up[0], cst[f]);
#pragma unroll
          for (int j = 1; j < D; ++j) e = fma2(bm[f][j], up[j], e);
        } else {
          u64 r2 = 0ull;
#pragma unroll
          for (int j = 0; j < D; ++j) {
            const u64 dx = add2(up[j], bm[f][j]);
            r2 = fma2(dx, dx, r2);
          }
          e = mul2(r2, cst[f]);
        }
        e = ex2x2(e);
        A[f] = fma2(e, al, A[f]);
#pragma unroll
        for (int j = 0; j < D; ++j) Q[f][j] = fma2(e, bp[j], Q[f][j]);
      }
    }
#pragma unroll
    for (int f = 0; f < F; ++f) {
      if (!ok[f]) continue;
      float lo, hi;
      upk(A[f], lo, hi);
      float v = lo + hi;
#pragma unroll
      for (int j = 0; j < D; ++j) {
        upk(Q[f][j], lo, hi);
        v = fmaf(c[f][j], lo + hi, v);
      }
      row[mf[f]] += v;
    }
  }
}

//   expanded: [a][b_0 ..][sg][c~_0 ..][h_q ..] (h_q = sg c_a c_b)     direct: [-mu_0 ..][lw][sg] (rest zero)
template <int D>
__device__ __forceinline__ void vj_stage_build(int64_t M, int64_t m0, bool expanded, const float* o, float gl2e,
                                               const float4* raw, u64* rec, int lane) {
  constexpr int RP = VjRbf<D>::kPairs;
  constexpr int KT = FastRec<D>::kTab;
  cp_async_wait_all();
  for (int i = lane; i < kWarpStage; i += 32) {
    const int64_t m = m0 + i;
    float mu[D], lw = -INFINITY, sg = 0.0f;
    if (m < M) {
      const float4 t0 = raw[i * KT];
      mu[0] = t0.x;
      mu[1] = t0.y;
      if (D == 2) {
        lw = t0.z;
        sg = t0.w;
      } else {
        mu[2] = t0.z;
        lw = t0.w;
        sg = raw[i * KT + 1].x;
      }
    } else {
#pragma unroll
      for (int j = 0; j < D; ++j) mu[j] = 0.0f;
    }
    u64 r[RP];
#pragma unroll
    for (int j = 0; j < RP; ++j) r[j] = 0ull;
    if (expanded) {
      float c[D], r2 = 0.0f;
#pragma unroll
      for (int j = 0; j < D; ++j) {
        c[j] = mu[j] - o[j];
        r2 = fmaf(c[j], c[j], r2);
      }
      const float a = fmaf(-gl2e, r2, lw);
      r[0] = pk(a, a);
#pragma unroll
      for (int j = 0; j < D; ++j) {
        const float b = 2.0f * gl2e * c[j], ct = sg * c[j];
        r[1 + j] = pk(b, b);
        r[D + 2 + j] = pk(ct, ct);
      }
#pragma unroll
      for (int ia = 0; ia < D; ++ia)
#pragma unroll
        for (int ib = 0; ib <= ia; ++ib) {
          const float h = sg * c[ia] * c[ib];
          r[2 * D + 2 + ia * (ia + 1) / 2 + ib] = pk(h, h);
        }
      r[D + 1] = pk(sg, sg);
    } else {
#pragma unroll
      for (int j = 0; j < D; ++j) r[j] = pk(-mu[j], -mu[j]);
      r[D] = pk(lw, lw);
      r[D + 1] = pk(sg, sg);
    }
    ulonglong2* dst = reinterpret_cast<ulonglong2*>(rec + (size_t)i * RP);
#pragma unroll
    for (int j = 0; j < RP / 2; ++j) dst[j] = make_ulonglong2(r[2 * j], r[2 * j + 1]);
  }
}

// sums of one pass at u (U) with v (V): S, G and H (expanded), or S, G and
// P = sum w phi ((x - mu) . v)(x - mu) in the first D entries of H (direct)
// (without SG, S and G are left alone: the caller has them from the recompute)
template <int D, int P, bool SG>
__device__ __forceinline__ void vj_stage_accumulate(const u64* rec, bool expanded, float gl2e, const u64 (&U)[P][D],
                                                    const u64 (&V)[P][D], u64 (&S)[P], u64 (&G)[P][D],
                                                    u64 (&H)[P][VjRbf<D>::kH]) {
  constexpr int NH = VjRbf<D>::kH;
  constexpr int RP = VjRbf<D>::kPairs;
  if (expanded) {
#pragma unroll 2
    for (int c = 0; c < kWarpStage; ++c) {
      const ulonglong2* q = reinterpret_cast<const ulonglong2*>(rec + (size_t)c * RP);
      u64 r[RP];
#pragma unroll
      for (int j = 0; j < RP / 2; ++j) {
        const ulonglong2 v = q[j];
        r[2 * j] = v.x;
        r[2 * j + 1] = v.y;
      }
#pragma unroll
      for (int i = 0; i < P; ++i) {
        u64 arg = fma2(r[1], U[i][0], r[0]);
#pragma unroll
        for (int j = 1; j < D; ++j) arg = fma2(r[1 + j], U[i][j], arg);
        const u64 e = ex2x2(arg);
        if (SG) {
          S[i] = fma2(r[D + 1], e, S[i]);
#pragma unroll
          for (int j = 0; j < D; ++j) G[i][j] = fma2(e, r[D + 2 + j], G[i][j]);
        }
#pragma unroll
        for (int q = 0; q < NH; ++q) H[i][q] = fma2(e, r[2 * D + 2 + q], H[i][q]);
      }
    }
  } else {
    const u64 ng = pk(-gl2e, -gl2e);
    for (int c = 0; c < kWarpStage; ++c) {
      const u64* r = rec + (size_t)c * RP;
#pragma unroll
      for (int i = 0; i < P; ++i) {
        u64 dx[D];
#pragma unroll
        for (int j = 0; j < D; ++j) dx[j] = add2(U[i][j], r[j]);
        u64 r2 = mul2(dx[0], dx[0]);
        u64 rv = mul2(dx[0], V[i][0]);
#pragma unroll
        for (int j = 1; j < D; ++j) {
          r2 = fma2(dx[j], dx[j], r2);
          rv = fma2(dx[j], V[i][j], rv);
        }
        const u64 we = mul2(r[D + 1], ex2x2(fma2(r2, ng, r[D])));   // w phi
        if (SG) S[i] = add2(S[i], we);
        const u64 wrv = mul2(we, rv);
#pragma unroll
        for (int j = 0; j < D; ++j) {
          if (SG) G[i][j] = fma2(we, dx[j], G[i][j]);
          H[i][j] = fma2(wrv, dx[j], H[i][j]);                 // sum w phi ((x - mu) . v)(x - mu)
        }
      }
    }
  }
}

// A tile's state x and cotangent g live in shared memory (xs, gs); every warp
// loads all of the tile's samples for a sweep, and each thread finishes its own
// one or two samples after it (samples threadIdx.x and + 128).
//
// CS > 1: a cluster of CS blocks shares the tile, each taking every CS-th group
// of centres; the blocks add up their sums through each other's shared memory
// and all finish every sample alike, so only the sums travel.
template <int D, bool GW, int CS>
__global__ void __launch_bounds__(VjRbf<D>::kW * 32, 3)
k_vjp_rbf_fast(TileArgs a, int kseg, const float* __restrict__ ckpt, const float* __restrict__ gT,
               float* __restrict__ g0, float* __restrict__ rows, int use_cache) {
  constexpr int W = VjRbf<D>::kW, K = VjRbf<D>::kK, P = K / 2, RP = VjRbf<D>::kPairs;
  constexpr int NS = VjRbf<D>::kSums, kTile = VjRbf<D>::kTile, KT = FastRec<D>::kTab, NH = VjRbf<D>::kH;
  constexpr int kOwn = (kTile + 32 * W - 1) / (32 * W);   // samples a thread finishes
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tile = (int)(blockIdx.x / CS), crank = (int)(blockIdx.x % CS);
  u64* wbuf = reinterpret_cast<u64*>(smem) + (size_t)warp * 2 * kWarpStage * RP;
  float* red = reinterpret_cast<float*>(smem);   // [W][NS][kTile], aliases the stages after a pass's last stage
  float4* red4 = reinterpret_cast<float4*>(smem);          // the recompute's: [W][kTile]
  float4* wraw = reinterpret_cast<float4*>(smem + vj_rbf_region0<D>()) + (size_t)warp * kWarpStage * KT;
  float* seg = reinterpret_cast<float*>(smem + vj_rbf_region0<D>() +
                                        (size_t)W * kWarpStage * KT * sizeof(float4));   // [kseg][D][kTile]
  const int64_t p0 = (int64_t)tile * kTile;
  const int64_t N = a.N, M = a.M;
  const float gamma = a.gamma, gl2e = gamma * kLog2e, eta = a.eta;
  // with the weight gradient a ragged tile visits every group: its empty slots sit at 0, where the expanded
  // sums can overflow, and what they then add to the row has to stay what it is without far groups
  const bool whole = GW && p0 + kTile > N;
  // weight gradient: this tile's row of rows[tiles][M + 1] (features in table order) and the sample terms after
  // the segment
  float* row = GW ? rows + (int64_t)tile * (M + 1) : nullptr;
  // the forward's S, G (cross-warp totals) at the segment's states: [kseg][1 + D][kTile]
  float* sgc = seg + (size_t)kseg * kTile * D;
  float* sm_gw = sgc + (use_cache ? (size_t)kseg * (1 + D) * kTile : 0);   // [kTile / 2][2D + 2] packed pairs
  float* xs = sm_gw + (GW ? (2 * D + 2) * kTile : 0);      // [D][kTile]
  float* gs = xs + D * kTile;                              // [D][kTile]
  float* ex = gs + D * kTile;                              // [NS][kTile], CS > 1: this block's sums
  NearSmem& ns = *reinterpret_cast<NearSmem*>(ex + (CS > 1 ? NS * kTile : 0));
  if (GW)   // this block's features
    for (int64_t g = crank; g * kGroup < M; g += CS)
      if (threadIdx.x < kGroup && g * kGroup + threadIdx.x < M) row[g * kGroup + threadIdx.x] = 0.0f;
  double gb = 0.0;   // the bias term of this thread's samples (one number for all of them: FP64)

  bool act[K];
#pragma unroll
  for (int k = 0; k < K; ++k) act[k] = p0 + k * 32 + lane < N;
  int64_t idx[kOwn];   // this thread's samples
  bool mine[kOwn];
#pragma unroll
  for (int h = 0; h < kOwn; ++h) {
    const int sm = threadIdx.x + h * 32 * W;
    mine[h] = sm < kTile && p0 + sm < N;
    idx[h] = mine[h] ? (int64_t)a.perm[p0 + sm] - a.perm_base : 0;
    if (sm < kTile)
#pragma unroll
      for (int j = 0; j < D; ++j) gs[j * kTile + sm] = mine[h] ? gT[idx[h] * D + j] : 0.0f;
  }

  // CS > 1: total of sum q (v: this block's) of sample sm over the cluster, in the blocks' order
  bool pending = false;   // the others may still read this block's sums
  auto publish = [&]() {
    if (CS > 1 && pending) cluster_wait();
  };
  auto exchange = [&]() {
    if (CS > 1) cluster_barrier();
  };
  auto release = [&]() {
    if (CS > 1) {
      cluster_arrive();
      pending = true;
    }
  };
  auto total = [&](int q, int sm) {
    float v = 0.0f;
#pragma unroll
    for (int r = 0; r < CS; ++r) {
      const float t = __uint_as_float(cluster_load(cluster_addr(&ex[q * kTile + sm], r)));
      v = r == 0 ? t : v + t;
    }
    return v;
  };

  const int nseg = a.T / kseg;
  for (int sgi = nseg - 1; sgi >= 0; --sgi) {
    const float* src = (sgi == 0 || ckpt == nullptr) ? a.x0 : ckpt + (int64_t)(sgi - 1) * N * D;
#pragma unroll
    for (int h = 0; h < kOwn; ++h) {
      const int sm = threadIdx.x + h * 32 * W;
      if (sm < kTile)
#pragma unroll
        for (int j = 0; j < D; ++j) xs[j * kTile + sm] = mine[h] ? src[idx[h] * D + j] : 0.0f;
    }
    const int pre = (sgi > 0 && ckpt == nullptr) ? sgi * kseg : 0;   // no checkpoints: recompute from x0
    for (int i = 0; i < pre + kseg; ++i) {
      if (i >= pre) {
#pragma unroll
        for (int h = 0; h < kOwn; ++h) {
          const int sm = threadIdx.x + h * 32 * W;
          if (sm < kTile)
#pragma unroll
            for (int j = 0; j < D; ++j) seg[((i - pre) * D + j) * kTile + sm] = xs[j * kTile + sm];
        }
        if (i == pre + kseg - 1) break;
      }
      __syncthreads();   // the states are visible, the reduction buffer is read
      // one forward step of the tile (every warp holds all its samples)
      float x[K][D], lo[D], hi[D], o[D];
#pragma unroll
      for (int k = 0; k < K; ++k)
#pragma unroll
        for (int j = 0; j < D; ++j) x[k][j] = xs[j * kTile + k * 32 + lane];
      const bool expanded = tile_frame<D, K>(x, act, gl2e, lo, hi, o);
      u64 U[P][D], S[P], G[P][D];
#pragma unroll
      for (int q = 0; q < P; ++q) {
#pragma unroll
        for (int j = 0; j < D; ++j) {
          U[q][j] = pk(x[2 * q][j] - o[j], x[2 * q + 1][j] - o[j]);
          G[q][j] = 0ull;
        }
        S[q] = 0ull;
      }
      for (int gb0 = 0; gb0 < a.ngroups; gb0 += kNearBatch) {
        if (gb0 > 0) __syncthreads();   // every warp has walked the batch before
        const int n = near_tile<D, W, K, CS>(a.box, a.ngroups, gb0, M, x, act, lo, hi, expanded, gl2e,
                                             whole ? kNearAll : kNearSums, ns, warp, lane, crank);
        near_sweep<D, P, false>(a.tab, M, gb0, NearWalk(ns, n, warp, W), expanded, o, gl2e, wraw, wbuf, lane, U, S, G);
      }
      __syncthreads();   // every warp has finished its centres before the reduction buffer overwrites the stages
      tile_put_sums<D, K>(S, G, red4 + warp * kTile, lane);
      __syncthreads();
      float4 acc[kOwn];
      publish();
#pragma unroll
      for (int h = 0; h < kOwn; ++h) {
        const int sm = threadIdx.x + h * 32 * W;
        acc[h] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (sm >= kTile) continue;
        acc[h] = red4[sm];
#pragma unroll
        for (int w = 1; w < W; ++w) add4(acc[h], red4[w * kTile + sm]);
        if (CS > 1) {
          ex[sm] = acc[h].x;
          ex[kTile + sm] = acc[h].y;
          ex[2 * kTile + sm] = acc[h].z;
          if (D == 3) ex[3 * kTile + sm] = acc[h].w;
        }
      }
      exchange();
#pragma unroll
      for (int h = 0; h < kOwn; ++h) {
        const int sm = threadIdx.x + h * 32 * W;
        if (sm >= kTile) continue;
        if (CS > 1) acc[h] = make_float4(total(0, sm), total(1, sm), total(2, sm), D == 3 ? total(3, sm) : 0.0f);
        if (use_cache && i >= pre) {   // for the Hessian-vector pass at the same state
          float* dst = sgc + (size_t)(i - pre) * (1 + D) * kTile + sm;
          dst[0] = acc[h].x;
          dst[kTile] = acc[h].y;
          dst[2 * kTile] = acc[h].z;
          if (D == 3) dst[3 * kTile] = acc[h].w;
        }
        float xo[1][D];
        const bool ao[1] = {mine[h]};
#pragma unroll
        for (int j = 0; j < D; ++j) xo[0][j] = xs[j * kTile + sm];
        tile_update<D, 1, false>(a, 0, p0, ao, xo, o, expanded, acc[h], 0, false, lane);
#pragma unroll
        for (int j = 0; j < D; ++j) xs[j * kTile + sm] = xo[0][j];
      }
      release();
    }
    for (int i = kseg - 1; i >= 0; --i) {
      __syncthreads();   // the segment's states, the cotangents (and the weight gradient's marks and terms) are done
      float x[K][D], g[K][D], lo[D], hi[D], o[D];
#pragma unroll
      for (int k = 0; k < K; ++k)
#pragma unroll
        for (int j = 0; j < D; ++j) {
          x[k][j] = seg[(i * D + j) * kTile + k * 32 + lane];
          g[k][j] = gs[j * kTile + k * 32 + lane];
        }
      const bool expanded = tile_frame<D, K>(x, act, gl2e, lo, hi, o);
      const bool have = use_cache && i < kseg - 1;   // S and G at this state from the recompute
      u64 U[P][D], V[P][D], S[P], G[P][D], H[P][NH];
#pragma unroll
      for (int q = 0; q < P; ++q) {
#pragma unroll
        for (int j = 0; j < D; ++j) {
          U[q][j] = pk(x[2 * q][j] - o[j], x[2 * q + 1][j] - o[j]);
          V[q][j] = pk(g[2 * q][j], g[2 * q + 1][j]);
          G[q][j] = 0ull;
        }
#pragma unroll
        for (int h = 0; h < NH; ++h) H[q][h] = 0ull;
        S[q] = 0ull;
      }
      for (int gb0 = 0; gb0 < a.ngroups; gb0 += kNearBatch) {
        if (gb0 > 0) __syncthreads();
        const int n = near_tile<D, W, K, CS>(a.box, a.ngroups, gb0, M, x, act, lo, hi, expanded, gl2e,
                                             whole ? kNearAll : kNearSums, ns, warp, lane, crank);
        NearWalk walk(ns, n, warp, W);
        int gi = walk.next();
        if (gi >= 0) {
          stage_prefetch<D>(a.tab, M, (int64_t)(gb0 + gi) * kWarpStage, wraw, lane);
          vj_stage_build<D>(M, (int64_t)(gb0 + gi) * kWarpStage, expanded, o, gl2e, wraw, wbuf, lane);
        }
        __syncwarp();
        for (int st = 0; gi >= 0; st ^= 1) {
          gi = walk.next();
          const int64_t mn = (int64_t)(gb0 + gi) * kWarpStage;
          const u64* cur = wbuf + (size_t)st * kWarpStage * RP;
          if (gi >= 0) stage_prefetch<D>(a.tab, M, mn, wraw, lane);
          if (have)
            vj_stage_accumulate<D, P, false>(cur, expanded, gl2e, U, V, S, G, H);
          else
            vj_stage_accumulate<D, P, true>(cur, expanded, gl2e, U, V, S, G, H);
          if (gi >= 0)
            vj_stage_build<D>(M, mn, expanded, o, gl2e, wraw, wbuf + (size_t)(st ^ 1) * kWarpStage * RP, lane);
          __syncwarp();
        }
      }
      __syncthreads();   // every warp has finished its centres before the reduction buffer overwrites the stages
      float* rw = red + (size_t)warp * NS * kTile;
#pragma unroll
      for (int q = 0; q < P; ++q) {
        float v0, v1;
        if (!have) {
          upk(S[q], v0, v1);
          rw[(2 * q) * 32 + lane] = v0;
          rw[(2 * q + 1) * 32 + lane] = v1;
#pragma unroll
          for (int j = 0; j < D; ++j) {
            upk(G[q][j], v0, v1);
            rw[(1 + j) * kTile + (2 * q) * 32 + lane] = v0;
            rw[(1 + j) * kTile + (2 * q + 1) * 32 + lane] = v1;
          }
        }
#pragma unroll
        for (int h = 0; h < NH; ++h) {   // H (direct: P in the first D)
          upk(H[q][h], v0, v1);
          rw[(1 + D + h) * kTile + (2 * q) * 32 + lane] = v0;
          rw[(1 + D + h) * kTile + (2 * q + 1) * 32 + lane] = v1;
        }
      }
      __syncthreads();
      float sums[kOwn][NS];
      publish();
#pragma unroll
      for (int h = 0; h < kOwn; ++h) {
        const int sm = threadIdx.x + h * 32 * W;
        if (sm >= kTile) continue;
#pragma unroll
        for (int q = 0; q < NS; ++q) {
          if (have && q <= D) {   // the recompute's totals at this state
            sums[h][q] = sgc[((size_t)i * (1 + D) + q) * kTile + sm];
            continue;
          }
          float v = red[q * kTile + sm];
#pragma unroll
          for (int w = 1; w < W; ++w) v += red[((size_t)w * NS + q) * kTile + sm];
          sums[h][q] = v;
          if (CS > 1) ex[q * kTile + sm] = v;
        }
      }
      exchange();
#pragma unroll
      for (int h = 0; h < kOwn; ++h) {
        const int sm = threadIdx.x + h * 32 * W;
        if (sm >= kTile) continue;
        if (CS > 1)
#pragma unroll
          for (int q = 0; q < NS; ++q)
            if (!(have && q <= D)) sums[h][q] = total(q, sm);
        const float(&sum)[NS] = sums[h];
        float xo[D], go[D];
#pragma unroll
        for (int j = 0; j < D; ++j) {
          xo[j] = seg[(i * D + j) * kTile + sm];
          go[j] = gs[j * kTile + sm];
        }
        const float Ss = sum[0];
        float shat, gsv[D], hv[D];
        if (expanded) {
          float u[D], u2 = 0.0f, uv = 0.0f;
#pragma unroll
          for (int j = 0; j < D; ++j) {
            u[j] = xo[j] - o[j];
            u2 = fmaf(u[j], u[j], u2);
            uv = fmaf(u[j], go[j], uv);
          }
          const float f = ex2_approx(-gl2e * u2);
          shat = f * Ss;
          float vG = 0.0f;   // K = sum e' (c . v) = v . G
#pragma unroll
          for (int j = 0; j < D; ++j) vG = fmaf(go[j], sum[1 + j], vG);
#pragma unroll
          for (int j = 0; j < D; ++j) {
            float Hv = 0.0f;   // Kc_j = (H v)_j, H from its lower triangle
#pragma unroll
            for (int i2 = 0; i2 < D; ++i2) {
              const int q = j >= i2 ? j * (j + 1) / 2 + i2 : i2 * (i2 + 1) / 2 + j;
              Hv = fmaf(sum[1 + D + q], go[i2], Hv);
            }
            const float usg = fmaf(u[j], Ss, -sum[1 + j]);                  // u S - G
            gsv[j] = -2.0f * gamma * (f * usg);
            const float m = fmaf(uv, usg, -fmaf(u[j], vG, -Hv));            // (u.v)(uS-G) - (u K - Kc)
            hv[j] = 4.0f * gamma * gamma * f * m - 2.0f * gamma * f * Ss * go[j];
          }
        } else {
          shat = Ss;
#pragma unroll
          for (int j = 0; j < D; ++j) {
            gsv[j] = -2.0f * gamma * sum[1 + j];
            hv[j] = 4.0f * gamma * gamma * sum[1 + D + j] - 2.0f * gamma * Ss * go[j];
          }
        }
        float d1, d2;
        sigmoid_d12(shat + a.bias, d1, d2);
        float gd = 0.0f;
#pragma unroll
        for (int j = 0; j < D; ++j) gd = fmaf(gsv[j], go[j], gd);
        if (GW) {   // the sample's weight-gradient terms, with g_{t+1}
          const float cA = mine[h] ? -eta * d2 * gd : 0.0f, cB = mine[h] ? -eta * d1 : 0.0f;
          float u[D], ug = 0.0f, f = 1.0f, u2 = 0.0f;
#pragma unroll
          for (int j = 0; j < D; ++j) {
            // direct form: o = 0; an empty slot sits at the origin, where phi / f <= 1 stays finite
            u[j] = mine[h] ? xo[j] - o[j] : 0.0f;
            ug = fmaf(u[j], go[j], ug);
            u2 = fmaf(u[j], u[j], u2);
          }
          if (expanded) f = ex2_approx(-gl2e * u2);
          gb += (double)cA;
#pragma unroll
          for (int j = 0; j < D; ++j) {
            GwTerms<D>::put(sm_gw, sm, j, u[j]);
            GwTerms<D>::put(sm_gw, sm, D + 1 + j, f * (2.0f * gamma * cB * go[j]));
          }
          GwTerms<D>::put(sm_gw, sm, D, f * fmaf(-2.0f * gamma * cB, ug, cA));
          GwTerms<D>::put(sm_gw, sm, 2 * D + 1, 0.0f);
        }
#pragma unroll
        for (int j = 0; j < D; ++j) gs[j * kTile + sm] = go[j] - eta * fmaf(d1, hv[j], d2 * gd * gsv[j]);
      }
      release();
      if (GW) {
        __syncthreads();   // the sample terms are visible
        for (int gb0 = 0; gb0 < a.ngroups; gb0 += kNearBatch) {
          if (gb0 > 0) __syncthreads();
          const int n = near_tile<D, W, K, CS>(a.box, a.ngroups, gb0, M, x, act, lo, hi, expanded, gl2e,
                                               whole ? kNearAll : kNearUnweighted, ns, warp, lane, crank);
          vj_gw_sweep<D, kTile>(a.tab, M, gb0, NearWalk(ns, n, warp, W), expanded, o, gl2e, sm_gw, row, lane);
        }
      }
    }
    __syncthreads();   // the cotangents and the last terms are read before the next segment
  }
  publish();           // no block leaves while another may read its sums
  if (GW && crank == 0) {
    double* sh = reinterpret_cast<double*>(smem);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) gb += __shfl_xor_sync(0xffffffffu, gb, off);
    if (lane == 0) sh[warp] = gb;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < W; ++w) gb += sh[w];
      row[M] = (float)gb;
    }
  }
  if (crank == 0)
#pragma unroll
    for (int h = 0; h < kOwn; ++h)
      if (mine[h])
#pragma unroll
        for (int j = 0; j < D; ++j) g0[idx[h] * D + j] = gs[j * kTile + threadIdx.x + h * 32 * W];
}

template <int D, bool GW, int CS>
static cudaError_t launch_vjp_shape(const TileArgs& a, int64_t tiles, int k, const float* ckpt, const float* gT,
                                    float* g0, float* rows, cudaStream_t st) {
  auto fn = k_vjp_rbf_fast<D, GW, CS>;
  // cache the recompute's S and G when the extra shared memory keeps as many blocks on an SM
  const size_t more = (2 * D + (CS > 1 ? VjRbf<D>::kSums : 0)) * VjRbf<D>::kTile * sizeof(float) + sizeof(NearSmem);
  const size_t smem0 = vj_rbf_smem<D>(k, GW, false) + more, smem1 = vj_rbf_smem<D>(k, GW, true) + more;
  int b0 = 0, b1 = 0;
  const bool fits = smem1 <= 227 * 1024;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(fits ? smem1 : smem0));
  if (e != cudaSuccess) return e;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b0, fn, VjRbf<D>::kW * 32, smem0);
  if (e == cudaSuccess && fits) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b1, fn, VjRbf<D>::kW * 32, smem1);
  if (e != cudaSuccess) return e;
  const int use_cache = b1 >= b0 && b1 > 0 ? 1 : 0;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3((unsigned)(tiles * CS));
  c.blockDim = dim3(VjRbf<D>::kW * 32);
  c.dynamicSmemBytes = use_cache ? smem1 : smem0;
  c.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CS;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  c.attrs = at;
  c.numAttrs = CS > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&c, fn, a, k, ckpt, gT, g0, rows, use_cache);
}

template <int D>
static cudaError_t launch_vjp_rbf_fast(const FieldArgs& fa, const float* x0, int64_t N, int T, float eta, int k,
                                       const float* ckpt, const float* gT, float* g0, float* rows, float* gw,
                                       float* gbias, void* ws, cudaStream_t st) {
  RbfOrder ord;
  cudaError_t e = rbf_order(D, fa.centres, fa.w, fa.M, x0, N, ws, &ord, st);
  if (e != cudaSuccess) return e;
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
  a.kck = 1;
  const int64_t tiles = vjp_rbf_fast_blocks(D, N);
  // Blocks per tile, measured with d/dw (M = 8192, T = 50, k = 5; forward and VJP in ms for 1, 2, 4, 8 blocks):
  // 59 tiles 21.1, 11.4, 8.1, 7.9; 117 12.6, 9.7, 7.8, 8.8; 235 22.0, 16.6, 14.4, 15.4; 782 tiles (M = 1000) 1.7,
  // 2.0, 3.0, 5.2.
  const int cs = tiles <= 114 ? 8 : (tiles <= 304 ? 4 : (tiles <= 456 ? 2 : 1));
  if (rows == nullptr) {
    if (cs == 8) return launch_vjp_shape<D, false, 8>(a, tiles, k, ckpt, gT, g0, nullptr, st);
    if (cs == 4) return launch_vjp_shape<D, false, 4>(a, tiles, k, ckpt, gT, g0, nullptr, st);
    if (cs == 2) return launch_vjp_shape<D, false, 2>(a, tiles, k, ckpt, gT, g0, nullptr, st);
    return launch_vjp_shape<D, false, 1>(a, tiles, k, ckpt, gT, g0, nullptr, st);
  }
  if (cs == 8) e = launch_vjp_shape<D, true, 8>(a, tiles, k, ckpt, gT, g0, rows, st);
  else if (cs == 4) e = launch_vjp_shape<D, true, 4>(a, tiles, k, ckpt, gT, g0, rows, st);
  else if (cs == 2) e = launch_vjp_shape<D, true, 2>(a, tiles, k, ckpt, gT, g0, rows, st);
  else e = launch_vjp_shape<D, true, 1>(a, tiles, k, ckpt, gT, g0, rows, st);
  if (e != cudaSuccess) return e;
  return sum_vjp_rows(rows, tiles, fa.M + 1, gw, gbias, st, ord.cperm);
}

int64_t vjp_rbf_fast_blocks(int d, int64_t N) {
  const int64_t tile = d == 2 ? VjRbf<2>::kTile : VjRbf<3>::kTile;
  return (N + tile - 1) / tile;
}

cudaError_t vjp_rbf_fast(int d, const FieldArgs& fa, const float* x0, int64_t N, int T, float eta, int k,
                         const float* ckpt, const float* gT, float* g0, float* rows, float* gw, float* gbias,
                         void* ws, cudaStream_t st) {
  if (d == 2) return launch_vjp_rbf_fast<2>(fa, x0, N, T, eta, k, ckpt, gT, g0, rows, gw, gbias, ws, st);
  if (d == 3) return launch_vjp_rbf_fast<3>(fa, x0, N, T, eta, k, ckpt, gT, g0, rows, gw, gbias, ws, st);
  return cudaErrorInvalidValue;
}

}  // namespace pdmp
