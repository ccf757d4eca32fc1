// Per-tile device code of the fast RBF morph (d = 2, 3), shared by the
// single-field launch (morph_rbf_fast.cu) and the batched launch (batch.cu).
//
#pragma once
#include "field.cuh"
#include "order.cuh"

namespace pdmp {

typedef unsigned long long u64;

__device__ __forceinline__ u64 pk(float lo, float hi) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void upk(u64 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
  u64 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
  u64 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
  u64 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// TF32 tensor-core pieces: round to TF32 (nearest, ties away), and
// D += A B for one m16n8k8 tile (A row-major 16 x 8, B column-major 8 x 8, FP32
// accumulate).  Fragments: with g = lane / 4 and t = lane % 4, a0 = A[g][t],
// a1 = A[g + 8][t], a2 = A[g][t + 4], a3 = A[g + 8][t + 4]; b0 = B[t][g],
// b1 = B[t + 4][g]; d0 = D[g][2t], d1 = D[g][2t + 1], d2 = D[g + 8][2t],
// d3 = D[g + 8][2t + 1].
__device__ __forceinline__ uint32_t tf32_rna(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ void mma_tf32(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ u64 ex2x2(u64 a) {
  float lo, hi;
  upk(a, lo, hi);
  return pk(ex2_approx(lo), ex2_approx(hi));
}
// 2^-a of both halves
__device__ __forceinline__ u64 ex2x2_neg(u64 a) {
  float lo, hi;
  upk(a, lo, hi);
  return pk(ex2_approx(-lo), ex2_approx(-hi));
}

// Tile shape: W warps per block (each summing over its share of M) and K
// samples per lane (even: f32x2 pairs).  The single-field launch uses
// W = 4, K = 10 (measured fastest on the 2-D fitted workload among K = 6..16,
// W = 2..8, unroll 1..4; 32-centre stages cost 1 % against 64 and make the
// groups that a tile can leave out smaller); the batched launch picks
// among a few shapes (autotuned).  Shapes with K > 8 need more than 128
// registers a thread and run 12 warps per SM, the others 16.
// The expanded exponent a_m + b_m . u carries a rounding error of about
// 2^-24 (|a_m| + |b_m . u|) <= 2^-24 3 g' R^2 for the features that matter
// (those within a few widths of the sample), i.e. a relative error of about
// 1.4e-6 in each feature at g' R^2 = 8; wider tiles take the direct form.
#ifndef PDMP_EXPAND_LIMIT
#define PDMP_EXPAND_LIMIT 8.0f
#endif
#ifndef PDMP_WARP_STAGE
#define PDMP_WARP_STAGE 32
#endif
#ifndef PDMP_FAST_UNROLL
#define PDMP_FAST_UNROLL 2
#endif
constexpr int kWarpStage = PDMP_WARP_STAGE;    // centres per warp per shared-memory stage
static_assert(kWarpStage == kGroup, "a stage is one group of ordered centres");
constexpr int kFastUnroll = PDMP_FAST_UNROLL;  // centres per unrolled inner iteration

template <int W, int K>
struct Shape {
  static_assert(K % 2 == 0, "samples per lane must be even (f32x2 pairs)");
  static constexpr int kWarps = W, kThreads = 32 * W, kK = K, kPairs = K / 2, kTile = 32 * K;
  static constexpr int kMinBlocks = (K > 8 ? 12 : 16) / W;   // warps per SM / warps per block
};

using FastShape = Shape<4, 10>;                // the single-field launch

template <int D>
struct FastRec {
  static constexpr int kPairs = 2 * D + 2;     // u64 pairs per staged centre
  static constexpr int kTab = D == 2 ? 1 : 2;  // float4s per centre in the table
};

// Shared memory of one tile: per warp, two stages of transformed records
// (aliased, after a step's last stage, by the cross-warp reduction buffer),
// then per warp the raw table entries of the stage being prefetched.
template <int D, int W>
__host__ __device__ constexpr size_t fast_bufs_bytes() {
  return (size_t)W * 2 * kWarpStage * FastRec<D>::kPairs * sizeof(u64);
}
template <int W, int K>
__host__ __device__ constexpr size_t fast_red_bytes() {
  return (size_t)W * (32 * K) * sizeof(float4);
}
template <int D, int W, int K>
__host__ __device__ constexpr size_t fast_region0_bytes() {
  return fast_bufs_bytes<D, W>() > fast_red_bytes<W, K>() ? fast_bufs_bytes<D, W>() : fast_red_bytes<W, K>();
}
template <int D, int W, int K>
__host__ __device__ constexpr size_t fast_smem_bytes() {
  return fast_region0_bytes<D, W, K>() + (size_t)W * kWarpStage * FastRec<D>::kTab * sizeof(float4);
}

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// One warp copies the table entries of centres [m0, m0 + kWarpStage) into
// its raw buffer (asynchronously; each lane copies the entries it later
// transforms).
template <int D>
__device__ __forceinline__ void stage_prefetch(const float4* __restrict__ tab, int64_t M, int64_t m0, float4* raw,
                                               int lane) {
  constexpr int KT = FastRec<D>::kTab;
  for (int i = lane; i < kWarpStage; i += 32) {
    const int64_t m = m0 + i;
    if (m < M)
#pragma unroll
      for (int q = 0; q < KT; ++q) cp_async16(raw + i * KT + q, tab + KT * m + q);
  }
  cp_async_commit();
}

// Waits for this lane's prefetched entries and writes the records of
// centres [m0, m0 + kWarpStage) into the warp's rec (kWarpStage x kPairs u64);
// the caller synchronises the warp before reading them.
//   expanded: [a a][b_0 b_0]..[b_{d-1} ..][sg sg][c~_0 c~_0]..  (c~ = sg (mu - o))
//   direct:   [-mu_0 -mu_0]..[-mu_{d-1} ..][lw lw][sg sg]
template <int D>
__device__ __forceinline__ void stage_build(int64_t M, int64_t m0, bool expanded, const float* o, float gl2e,
                                            const float4* raw, u64* rec, int lane) {
  constexpr int RP = FastRec<D>::kPairs;
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
    if (expanded) {
      float c[D], r2 = 0.0f;
#pragma unroll
      for (int j = 0; j < D; ++j) {
        c[j] = mu[j] - o[j];
        r2 = fmaf(c[j], c[j], r2);
      }
      float a = fmaf(-gl2e, r2, lw);
      r[0] = pk(a, a);
#pragma unroll
      for (int j = 0; j < D; ++j) {
        float b = 2.0f * gl2e * c[j];
        r[1 + j] = pk(b, b);
        float ct = sg * c[j];
        r[D + 2 + j] = pk(ct, ct);
      }
      r[D + 1] = pk(sg, sg);
    } else {
#pragma unroll
      for (int j = 0; j < D; ++j) r[j] = pk(-mu[j], -mu[j]);
      r[D] = pk(lw, lw);
      r[D + 1] = pk(sg, sg);
#pragma unroll
      for (int j = D + 2; j < RP; ++j) r[j] = 0ull;
    }
    ulonglong2* dst = reinterpret_cast<ulonglong2*>(rec + (size_t)i * RP);
#pragma unroll
    for (int j = 0; j < RP / 2; ++j) dst[j] = make_ulonglong2(r[2 * j], r[2 * j + 1]);
  }
}

// Arguments of one tile: a run of 256 (32 K) consecutive sorted positions
// [p0, min(p0 + tile, p_end)) of one field's samples.  perm maps a sorted
// position to a sample index; the sample's index in x0 / xT / ckpt / traj /
// steps is perm[p] - perm_base, and those arrays hold N samples.
struct TileArgs {
  const float4* tab;     // centre table in the order of rbf_order
  const float4* box;     // its groups' boxes
  int ngroups;
  int64_t M;
  float gamma, bias, eta;
  int T;
  const float* x0;
  const int32_t* perm;
  int64_t perm_base;
  int64_t N;
  float* xT;
  float* ckpt;
  int kck;
  float* traj;
  float* steps;
  float* s_out;   // optional: the logit s(x_{T-1}) of the last step, per sample
  float* g_out;   // optional: grad c(x_{T-1}) of the last step, per sample (d values)
};

// Bounding box of the tile's active samples (identical in every warp: each
// warp holds all of them); its centre o is the origin of the expanded form,
// which the step uses only while g' R^2 <= PDMP_EXPAND_LIMIT (R the
// half-diagonal).
template <int D, int K>
__device__ __forceinline__ bool tile_frame(const float (&x)[K][D], const bool (&act)[K], float gl2e, float (&lo)[D],
                                           float (&hi)[D], float (&o)[D]) {
#pragma unroll
  for (int j = 0; j < D; ++j) { lo[j] = INFINITY; hi[j] = -INFINITY; }
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (act[k])
#pragma unroll
      for (int j = 0; j < D; ++j) { lo[j] = fminf(lo[j], x[k][j]); hi[j] = fmaxf(hi[j], x[k][j]); }
  float R2 = 0.0f;
#pragma unroll
  for (int j = 0; j < D; ++j) {
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
      lo[j] = fminf(lo[j], __shfl_xor_sync(0xffffffffu, lo[j], s));
      hi[j] = fmaxf(hi[j], __shfl_xor_sync(0xffffffffu, hi[j], s));
    }
    o[j] = 0.5f * (lo[j] + hi[j]);
    float h = 0.5f * (hi[j] - lo[j]);
    R2 = fmaf(h, h, R2);
  }
  const bool expanded = (gl2e * R2 <= PDMP_EXPAND_LIMIT) && (o[0] == o[0]);
  if (!expanded)
#pragma unroll
    for (int j = 0; j < D; ++j) o[j] = 0.0f;
  return expanded;
}

// ------------------------------------------------------------- near groups
// With y = g' d^2, d the distance between a group's box and the tile's, the
// group's terms of s are at most 2^(lw_max - y) for every sample of the tile.  A
// group is far, and left out, in two cases.
//
// (1) Its terms are exactly zero: the exponents the kernels form are at most
// lw_max - y (the expanded form's + g' R^2, its factor f = 2^(-g' |u|^2) taken
// out), and ex2.approx.ftz returns 0 below -126.  One unit more covers the
// rounding of the exponents and of this test.
//
// (2) All far groups together are below FP32's rounding of the sums.  Every
// group's strongest centre mu* bounds one term of the sums from below for every
// sample of the tile: of s by 2^(lw* - g' dmax^2), of grad s by that times the
// distance, sqrt(g') dmin; let ref be the largest of the latter (at most the
// largest of the former).  Beyond y = 1 a feature's terms of s, grad s and Hess
// s (2 gamma (1 + 2 gamma d^2) relative to s's) fall with d, so that with
//   lw_max - y + log2(1 + 2 gamma d^2) < log2(ref) - (30 + log2 M)
// the M features at most that are left out add up to less than 2^-30 of a term
// that is summed: 1/64 of the rounding error that this term alone brings
// (FP32's half ulp, 2^-25), whatever cancels.  Not used where a feature stands
// without its weight or is an output itself (the weight gradient).
//
// A tile with a sample that is not finite has no far groups (its sums must
// reach it).
//
// The near groups of a sweep are listed in shared memory by all warps of the
// block together, kNearBatch groups (65,536 centres) at a time; every warp then
// walks the entries that are its own.
constexpr int kNearBatch = 2048;

struct NearSmem {
  uint32_t words[kNearBatch / 32];   // a bit per group of the batch
  float refs[16];                    // the warps' largest ref
  float state[8];                    // the tile's box and limits, for batches after the first
  uint16_t list[kNearBatch];         // the near groups, relative to the batch
};

// A warp's share of the list: entries own, own + stride, ...
struct NearWalk {
  const uint16_t* list;
  int n, i, stride;
  __device__ __forceinline__ NearWalk(const NearSmem& s, int count, int own, int st)
      : list(s.list), n(count), i(own), stride(st) {}
  // the next one, or -1 (the same in every lane)
  __device__ __forceinline__ int next() {
    if (i >= n) return -1;
    const int g = list[i];
    i += stride;
    return g;
  }
};

// Lists the groups of the range g0 + [0, kNearBatch) below ngroups for which
// near(g) holds, in order, and returns how many; W warps, two block barriers
// (the second makes the list visible).
template <int W, typename F>
__device__ __forceinline__ int near_list(NearSmem& s, int g0, int ngroups, int warp, int lane, F near) {
  const int cnt = ngroups - g0 < kNearBatch ? ngroups - g0 : kNearBatch, nw = (cnt + 31) / 32;
#pragma unroll 2
  for (int q = warp; q < nw; q += W) {
    const int g = q * 32 + lane;
    const uint32_t m = __ballot_sync(0xffffffffu, g < cnt && near(g0 + g));
    if (lane == 0) s.words[q] = m;
  }
  __syncthreads();
  // exclusive prefix of the words' counts: lane l holds words l and l + 32
  uint32_t c0 = lane < nw ? __popc(s.words[lane]) : 0u, c1 = lane + 32 < nw ? __popc(s.words[lane + 32]) : 0u;
  const uint32_t n0 = c0, n1 = c1;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t0 = __shfl_up_sync(0xffffffffu, c0, o), t1 = __shfl_up_sync(0xffffffffu, c1, o);
    if (lane >= o) {
      c0 += t0;
      c1 += t1;
    }
  }
  const uint32_t first = __shfl_sync(0xffffffffu, c0, 31), total = first + __shfl_sync(0xffffffffu, c1, 31);
  c0 -= n0;
  c1 += first - n1;
  for (int q = warp; q < nw; q += W) {
    const uint32_t m = s.words[q], at = __shfl_sync(0xffffffffu, q < 32 ? c0 : c1, q & 31);
    if (m >> lane & 1u) s.list[at + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(q * 32 + lane);
  }
  __syncthreads();
  return (int)total;
}

// what near_tile lists
enum NearRule { kNearSums, kNearUnweighted, kNearAll };

// Lists the groups of batch g0 that are near the tile's box [lo, hi] (of x, the
// same in every warp).  kNearSums: rules (1) and (2); kNearUnweighted: rule (1)
// for sums in which phi stands without its weight; kNearAll: every group.  CS >
// 1: only every CS-th group, those of block crank of a cluster.  The
// first batch (g0 = 0) computes the limits; later ones take them, and the box,
// from shared memory.  A block barrier must separate it from the walks before.
template <int D, int W, int K, int CS = 1>
__device__ __forceinline__ int near_tile(const float4* __restrict__ box, int ngroups, int g0, int64_t M,
                                         const float (&x)[K][D], const bool (&act)[K], float (&lo)[D], float (&hi)[D],
                                         bool expanded, float gl2e, NearRule rule, NearSmem& s, int warp, int lane,
                                         int crank = 0) {
  float lim1, lim2;
  if (g0 == 0) {
    float ref = -INFINITY;
    if (rule == kNearSums) {
      // of few groups every warp goes over all (no exchange), of many over its share
      const bool share = ngroups > 64;
      for (int g = (share ? warp * 32 : 0) + lane; g < ngroups; g += (share ? W : 1) * 32) {
        const float4 b = box[kGroupBox * g + 2];
        const float mu[3] = {b.x, b.y, b.z};
        float dmin2 = 0.0f, dmax2 = 0.0f;
#pragma unroll
        for (int j = 0; j < D; ++j) {
          const float gap = fmaxf(0.0f, fmaxf(mu[j] - hi[j], lo[j] - mu[j]));
          const float reach = fmaxf(hi[j] - mu[j], mu[j] - lo[j]);
          dmin2 = fmaf(gap, gap, dmin2);
          dmax2 = fmaf(reach, reach, dmax2);
        }
        ref = fmaxf(ref, fmaf(-gl2e, dmax2, b.w) + 0.5f * lg2_approx(fminf(1.0f, gl2e * dmin2)));
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) ref = fmaxf(ref, __shfl_xor_sync(0xffffffffu, ref, o));
      if (share) {
        if (lane == 0) s.refs[warp] = ref;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < W; ++w) ref = fmaxf(ref, s.refs[w]);
      }
    }
    float R2 = 0.0f;
    bool odd = false;
#pragma unroll
    for (int j = 0; j < D; ++j) {
      const float h = 0.5f * (hi[j] - lo[j]);
      R2 = fmaf(h, h, R2);
    }
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
      for (int j = 0; j < D; ++j) odd = odd || (act[k] && !(fabsf(x[k][j]) < INFINITY));
    odd = __any_sync(0xffffffffu, odd);
    lim1 = odd || rule == kNearAll ? INFINITY : 127.0f + (expanded ? gl2e * R2 : 0.0f);
    lim2 = odd || rule != kNearSums ? INFINITY : 30.0f + lg2_approx((float)M) - ref;
    if (ngroups > kNearBatch && threadIdx.x == 0) {
#pragma unroll
      for (int j = 0; j < D; ++j) {
        s.state[j] = lo[j];
        s.state[3 + j] = hi[j];
      }
      s.state[6] = lim1;
      s.state[7] = lim2;
    }
  } else {
#pragma unroll
    for (int j = 0; j < D; ++j) {
      lo[j] = s.state[j];
      hi[j] = s.state[3 + j];
    }
    lim1 = s.state[6];
    lim2 = s.state[7];
  }
  return near_list<W>(s, g0, ngroups, warp, lane, [&](int g) {
    if (CS > 1 && (g & (CS - 1)) != crank) return false;
    const float4 b0 = box[kGroupBox * g], b1 = box[kGroupBox * g + 1];
    const float blo[3] = {b0.x, b0.y, b0.z}, bhi[3] = {b1.x, b1.y, b1.z};
    float d2 = 0.0f;
#pragma unroll
    for (int j = 0; j < D; ++j) {
      const float gap = fmaxf(0.0f, fmaxf(blo[j] - hi[j], lo[j] - bhi[j]));
      d2 = fmaf(gap, gap, d2);
    }
    const float y = gl2e * d2, below = y - (rule == kNearUnweighted ? fmaxf(b0.w, 0.0f) : b0.w);
    // 2 gamma d^2 = 2 ln 2 y
    return !(below > lim1 || (y > 1.0f && below - lg2_approx(fmaf(1.38629436f, y, 1.0f)) > lim2));
  });
}

// Adds the kWarpStage staged records rec to the pair sums S, G of this lane's
// samples (U: the samples relative to the origin, packed in pairs).
template <int D, int P>
__device__ __forceinline__ void stage_accumulate(const u64* rec, bool expanded, float gl2e, const u64 (&U)[P][D],
                                                 u64 (&S)[P], u64 (&G)[P][D]) {
  constexpr int RP = FastRec<D>::kPairs;
  if (expanded) {
#pragma unroll (P <= 2 ? 4 : kFastUnroll)
    for (int c = 0; c < kWarpStage; ++c) {
      const ulonglong2* q = reinterpret_cast<const ulonglong2*>(rec + (size_t)c * RP);
      u64 r[RP];
#pragma unroll
      for (int j = 0; j < RP / 2; ++j) {
        ulonglong2 v = q[j];
        r[2 * j] = v.x;
        r[2 * j + 1] = v.y;
      }
      // phased: the P arguments, their ex2, then each sum over the P pairs, so
      // that consecutive packed FMAs share the record's operand (1.2 % faster
      // than pair by pair, measured; identical results)
      u64 e[P];
#pragma unroll
      for (int i = 0; i < P; ++i) e[i] = fma2(r[1], U[i][0], r[0]);
#pragma unroll
      for (int j = 1; j < D; ++j)
#pragma unroll
        for (int i = 0; i < P; ++i) e[i] = fma2(r[1 + j], U[i][j], e[i]);
#pragma unroll
      for (int i = 0; i < P; ++i) e[i] = ex2x2(e[i]);
#pragma unroll
      for (int i = 0; i < P; ++i) S[i] = fma2(r[D + 1], e[i], S[i]);
#pragma unroll
      for (int j = 0; j < D; ++j)
#pragma unroll
        for (int i = 0; i < P; ++i) G[i][j] = fma2(e[i], r[D + 2 + j], G[i][j]);
    }
  } else {
    const u64 ng = pk(-gl2e, -gl2e);
    auto one = [&](int c) {
      const u64* r = rec + (size_t)c * RP;
#pragma unroll
      for (int i = 0; i < P; ++i) {
        u64 dx[D];
#pragma unroll
        for (int j = 0; j < D; ++j) dx[j] = add2(U[i][j], r[j]);
        u64 r2 = mul2(dx[0], dx[0]);
#pragma unroll
        for (int j = 1; j < D; ++j) r2 = fma2(dx[j], dx[j], r2);
        const u64 we = mul2(r[D + 1], ex2x2(fma2(r2, ng, r[D])));
        S[i] = add2(S[i], we);
#pragma unroll
        for (int j = 0; j < D; ++j) G[i][j] = fma2(we, dx[j], G[i][j]);
      }
    };
    if constexpr (P <= 2) {   // few pairs: more centres in flight
#pragma unroll 4
      for (int c = 0; c < kWarpStage; ++c) one(c);
    } else {
      for (int c = 0; c < kWarpStage; ++c) one(c);
    }
  }
}

// The direct form about the tile centre o for tiles too wide for the expanded
// one (the batched launch's tiles): x - mu per feature in coordinates scaled
// by sqrt(g'), so that -log2 e = |x' - mu'|^2 - log2|w| takes d FMAs from the
// record's -log2|w|, and the sign rides in S's FMA:
//   S = sum sg e,  G' = sum sg e (mu - o),  so  sum w phi (x - mu) = u S - G'
// with u = x - o: 3d + 1 packed operations per sample pair and feature
// (the direct form about 0 takes 3d + 3).  Records:
//   [-c'_0 -c'_0]..[-c'_{d-1} ..][-lw -lw][sg sg][c~_0 c~_0]..
//   (c = mu - o, c' = sqrt(g') c, c~ = sg c)
template <int D>
__device__ __forceinline__ void stage_build_origin(int64_t M, int64_t m0, const float* o, float gl2e,
                                                   const float4* raw, u64* rec, int lane) {
  constexpr int RP = FastRec<D>::kPairs;
  constexpr int KT = FastRec<D>::kTab;
  const float sc = sqrtf(gl2e);
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
      for (int j = 0; j < D; ++j) mu[j] = o[j];
    }
    u64 r[RP];
#pragma unroll
    for (int j = 0; j < D; ++j) {
      const float c = mu[j] - o[j], cs = -sc * c, ct = sg * c;
      r[j] = pk(cs, cs);
      r[D + 2 + j] = pk(ct, ct);
    }
    r[D] = pk(-lw, -lw);
    r[D + 1] = pk(sg, sg);
    ulonglong2* dst = reinterpret_cast<ulonglong2*>(rec + (size_t)i * RP);
#pragma unroll
    for (int j = 0; j < RP / 2; ++j) dst[j] = make_ulonglong2(r[2 * j], r[2 * j + 1]);
  }
}

// U holds sqrt(g') (x - o); S, G' as above
template <int D, int P>
__device__ __forceinline__ void stage_accumulate_origin(const u64* rec, const u64 (&U)[P][D], u64 (&S)[P],
                                                        u64 (&G)[P][D]) {
  constexpr int RP = FastRec<D>::kPairs;
  auto one = [&](int c) {
    const u64* r = rec + (size_t)c * RP;
#pragma unroll
    for (int i = 0; i < P; ++i) {
      u64 q = r[D];
#pragma unroll
      for (int j = 0; j < D; ++j) {
        const u64 dx = add2(U[i][j], r[j]);
        q = fma2(dx, dx, q);
      }
      const u64 e = ex2x2_neg(q);
      S[i] = fma2(r[D + 1], e, S[i]);
#pragma unroll
      for (int j = 0; j < D; ++j) G[i][j] = fma2(e, r[D + 2 + j], G[i][j]);
    }
  };
  if constexpr (P <= 2) {
#pragma unroll 4
    for (int c = 0; c < kWarpStage; ++c) one(c);
  } else {
    for (int c = 0; c < kWarpStage; ++c) one(c);
  }
}

// Loads the tile's samples (sorted positions [p0, p_end)).
template <int D, int K>
__device__ __forceinline__ void tile_load(const TileArgs& a, int64_t p0, int64_t p_end, int lane, float (&x)[K][D],
                                          bool (&act)[K]) {
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int64_t p = p0 + k * 32 + lane;
    act[k] = p < p_end;
    const int64_t n = act[k] ? (int64_t)a.perm[p] - a.perm_base : 0;
#pragma unroll
    for (int j = 0; j < D; ++j) x[k][j] = act[k] ? a.x0[n * D + j] : 0.0f;
  }
}

// End of step t for sample k of this lane: the Euler update of Eq. (1) from
// the totals acc = (S, G) of its sums; the writer (one warp of the tile) also
// writes the trace and the last logit and gradient.
template <int D, int K, bool TRACE>
__device__ __forceinline__ void tile_update(const TileArgs& a, int t, int64_t p0, const bool (&act)[K],
                                            float (&x)[K][D], const float (&o)[D], bool expanded, const float4& acc,
                                            int k, bool writer, int lane) {
  const int64_t N = a.N;
  const float gamma = a.gamma, bias = a.bias, eta = a.eta;
  const int T = a.T;
  const float gl2e = gamma * kLog2e;
  const float Ssum = acc.x, Gs[3] = {acc.y, acc.z, acc.w};
  float shat, ghat[D];
  if (expanded) {
    float u[D], u2 = 0.0f;
#pragma unroll
    for (int j = 0; j < D; ++j) {
      u[j] = x[k][j] - o[j];
      u2 = fmaf(u[j], u[j], u2);
    }
    const float f = ex2_approx(-gl2e * u2);
    shat = f * Ssum;
#pragma unroll
    for (int j = 0; j < D; ++j) ghat[j] = f * fmaf(u[j], Ssum, -Gs[j]);
  } else {
    shat = Ssum;
#pragma unroll
    for (int j = 0; j < D; ++j) ghat[j] = Gs[j];
  }
  float d1, d2;
  sigmoid_d12(shat + bias, d1, d2);
  const float c = -eta * d1;
  const int64_t p = p0 + k * 32 + lane;
  const bool own = act[k] && writer;
  const bool last_out = t == T - 1 && (a.s_out != nullptr || a.g_out != nullptr);
  const int64_t n = (own && (TRACE || last_out)) ? (int64_t)a.perm[p] - a.perm_base : 0;
  if (own && a.s_out != nullptr && t == T - 1) a.s_out[n] = shat + bias;
  if (own && a.g_out != nullptr && t == T - 1)
#pragma unroll
    for (int j = 0; j < D; ++j) a.g_out[n * D + j] = d1 * (-2.0f * gamma * ghat[j]);
#pragma unroll
  for (int j = 0; j < D; ++j) {
    const float inc = __fmul_rn(c, -2.0f * gamma * ghat[j]);
    if (TRACE && act[k] && writer) {
      a.traj[((int64_t)t * N + n) * D + j] = x[k][j];
      a.steps[((int64_t)t * N + n) * D + j] = inc;
    }
    x[k][j] = __fadd_rn(x[k][j], inc);
  }
}

// The checkpoint after step t, if one is due (called by the writer warp).
template <int D, int K>
__device__ __forceinline__ void tile_checkpoint(const TileArgs& a, int t, int64_t p0, const bool (&act)[K],
                                                const float (&x)[K][D], int lane) {
  if (a.ckpt == nullptr || (t + 1) % a.kck != 0) return;
  float* dst = a.ckpt + (int64_t)((t + 1) / a.kck - 1) * a.N * D;
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (act[k]) {
      const int64_t n = (int64_t)a.perm[p0 + k * 32 + lane] - a.perm_base;
#pragma unroll
      for (int j = 0; j < D; ++j) dst[n * D + j] = x[k][j];
    }
}

// Writes one warp's sums of the tile's samples to dst (32 K float4s).
template <int D, int K>
__device__ __forceinline__ void tile_put_sums(const u64 (&S)[K / 2], const u64 (&G)[K / 2][D], float4* dst, int lane) {
#pragma unroll
  for (int i = 0; i < K / 2; ++i) {
    float s0, s1, g0[D], g1[D];
    upk(S[i], s0, s1);
#pragma unroll
    for (int j = 0; j < D; ++j) upk(G[i][j], g0[j], g1[j]);
    dst[(2 * i) * 32 + lane] = make_float4(s0, g0[0], g0[1], D == 3 ? g0[D - 1] : 0.0f);
    dst[(2 * i + 1) * 32 + lane] = make_float4(s1, g1[0], g1[1], D == 3 ? g1[D - 1] : 0.0f);
  }
}

// ... or adds them to what is there (its own: a lane adds to what it wrote).
template <int D, int K>
__device__ __forceinline__ void tile_add_sums(const u64 (&S)[K / 2], const u64 (&G)[K / 2][D], float4* dst, int lane) {
#pragma unroll
  for (int i = 0; i < K / 2; ++i) {
    float s[2], g0[2], g1[2], g2[2] = {0.0f, 0.0f};
    upk(S[i], s[0], s[1]);
    upk(G[i][0], g0[0], g0[1]);
    upk(G[i][1], g1[0], g1[1]);
    if (D == 3) upk(G[i][D - 1], g2[0], g2[1]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float4& d = dst[(2 * i + h) * 32 + lane];
      d = make_float4(d.x + s[h], d.y + g0[h], d.z + g1[h], d.w + g2[h]);
    }
  }
}

__device__ __forceinline__ void add4(float4& acc, const float4& b) {
  acc.x += b.x;
  acc.y += b.y;
  acc.z += b.z;
  acc.w += b.w;
}

// End of step t: the warps' partial sums are added in a fixed order (every
// warp computes the same totals), then the update of every sample.  Begins and
// ends with a block barrier (the reduction buffer aliases the stage buffers).
template <int D, int W, int K, bool TRACE>
__device__ __forceinline__ void tile_finish_step(const TileArgs& a, int t, int64_t p0, const bool (&act)[K],
                                                 float (&x)[K][D], const float (&o)[D], bool expanded,
                                                 const u64 (&S)[K / 2], const u64 (&G)[K / 2][D], float4* red,
                                                 int warp, int lane) {
  constexpr int kTile = 32 * K;
  __syncthreads();   // every warp has finished its centres before the reduction buffer overwrites the stages
  tile_put_sums<D, K>(S, G, red + warp * kTile, lane);
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) {
    float4 acc = red[k * 32 + lane];
#pragma unroll
    for (int w = 1; w < W; ++w) add4(acc, red[w * kTile + k * 32 + lane]);
    tile_update<D, K, TRACE>(a, t, p0, act, x, o, expanded, acc, k, warp == 0, lane);
  }
  __syncthreads();   // every warp has read the reduction buffer before the next step rebuilds the stages
  if (warp == 0) tile_checkpoint<D, K>(a, t, p0, act, x, lane);
}

// Writes x_T (and the trace's last state) of the tile's samples.
template <int D, int K, bool TRACE>
__device__ __forceinline__ void tile_store(const TileArgs& a, int64_t p0, const bool (&act)[K],
                                           const float (&x)[K][D], int warp, int lane) {
  if (warp == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k)
      if (act[k]) {
        const int64_t n = (int64_t)a.perm[p0 + k * 32 + lane] - a.perm_base;
#pragma unroll
        for (int j = 0; j < D; ++j) {
          if (a.xT) a.xT[n * D + j] = x[k][j];
          if (TRACE) a.traj[((int64_t)a.T * a.N + n) * D + j] = x[k][j];
        }
      }
  }
  __syncthreads();   // the next tile of this block reuses the shared memory
}

// The sums S, G over the near groups of one walk, double-buffered through the
// warp's two stages.  ORIGIN: see fast_tile.
template <int D, int P, bool ORIGIN>
__device__ __forceinline__ void near_sweep(const float4* __restrict__ tab, int64_t M, int g0, NearWalk walk,
                                           bool expanded, const float (&o)[D], float gl2e, float4* wraw, u64* wbuf,
                                           int lane, const u64 (&U)[P][D], u64 (&S)[P], u64 (&G)[P][D]) {
  constexpr int RP = FastRec<D>::kPairs;
  int g = walk.next();
  if (g < 0) return;
  u64* cur = wbuf;
  u64* nxt = wbuf + (size_t)kWarpStage * RP;
  stage_prefetch<D>(tab, M, (int64_t)(g0 + g) * kWarpStage, wraw, lane);
  if (ORIGIN && !expanded)
    stage_build_origin<D>(M, (int64_t)(g0 + g) * kWarpStage, o, gl2e, wraw, cur, lane);
  else
    stage_build<D>(M, (int64_t)(g0 + g) * kWarpStage, expanded, o, gl2e, wraw, cur, lane);
  __syncwarp();
  do {
    g = walk.next();
    const int64_t mn = (int64_t)(g0 + g) * kWarpStage;
    if (g >= 0) stage_prefetch<D>(tab, M, mn, wraw, lane);
    if (ORIGIN && !expanded) {
      stage_accumulate_origin<D, P>(cur, U, S, G);
      if (g >= 0) stage_build_origin<D>(M, mn, o, gl2e, wraw, nxt, lane);
    } else {
      stage_accumulate<D, P>(cur, expanded, gl2e, U, S, G);
      if (g >= 0) stage_build<D>(M, mn, expanded, o, gl2e, wraw, nxt, lane);
    }
    __syncwarp();
    u64* const swap = cur;
    cur = nxt;
    nxt = swap;
  } while (g >= 0);
}

// A tile's near groups are dealt out to kLeaves<W, K> partial sums, the totals
// adding them in order.  Tiles of 320 samples have one per warp.  128-sample
// tiles have 16 whatever the number of warps, so that a launch of few tiles
// may spread a tile over a cluster of 2 or 4 blocks (CS) with the same result
// bit for bit as one block of 4 warps that takes 4 leaves each.
template <int W, int K>
__host__ __device__ constexpr int tile_leaves() { return K == 4 ? 16 : W; }

template <int D, int W, int K, int CS = 1>
__host__ __device__ constexpr size_t tile_leaf_bytes() {
  return tile_leaves<W, K>() == W ? 0
                                  : (size_t)tile_leaves<W, K>() / CS * (CS > 1 ? 2 : 1) * (32 * K) * sizeof(float4);
}
// (with NearSmem at the end)
template <int D, int W, int K, int CS = 1>
__host__ __device__ constexpr size_t tile_smem_bytes() {
  return fast_smem_bytes<D, W, K>() + tile_leaf_bytes<D, W, K, CS>() +
         (tile_leaves<W, K>() == W ? 0 : (size_t)32 * K * D * sizeof(float)) + sizeof(NearSmem);
}

// ORIGIN: tiles too wide for the expanded form take the direct form about the
// tile centre (stage_build_origin) instead of the one about 0.  The
// single-field launch keeps the latter: there nearly every tile is expanded,
// and the kernel compiled with both forms ran 6 % slower on such tiles.
// CS > 1: the tile is shared by the blocks of a cluster, this one of rank
// crank; the launch is not persistent.
template <int D, int W, int K, bool TRACE, bool ORIGIN = false, int CS = 1>
__device__ __forceinline__ void fast_tile(const TileArgs& a, int64_t p0, int64_t p_end, unsigned char* smem,
                                          int crank = 0) {
  constexpr int RP = FastRec<D>::kPairs;
  constexpr int P = K / 2;
  constexpr int KT = FastRec<D>::kTab;
  constexpr int L = tile_leaves<W, K>(), WT = W * CS, kTile = 32 * K;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // each warp has its own stage buffers
  u64* wbuf = reinterpret_cast<u64*>(smem) + (size_t)warp * 2 * kWarpStage * RP;
  float4* red = reinterpret_cast<float4*>(smem);   // aliases the stage buffers after a step's last stage
  float4* wraw = reinterpret_cast<float4*>(smem + fast_region0_bytes<D, W, K>()) + (size_t)warp * kWarpStage * KT;
  float4* leaves = reinterpret_cast<float4*>(smem + fast_smem_bytes<D, W, K>());
  float* xs = reinterpret_cast<float*>(smem + fast_smem_bytes<D, W, K>() + tile_leaf_bytes<D, W, K, CS>());
  NearSmem& ns = *reinterpret_cast<NearSmem*>(smem + tile_smem_bytes<D, W, K, CS>() - sizeof(NearSmem));
  const float gl2e = a.gamma * kLog2e;
  const bool writer = warp == 0 && crank == 0;

  float x[K][D];
  bool act[K];
  tile_load<D, K>(a, p0, p_end, lane, x, act);

  for (int t = 0; t < a.T; ++t) {
    float lo[D], hi[D], o[D];
    const bool expanded = tile_frame<D, K>(x, act, gl2e, lo, hi, o);
    if (ORIGIN && !expanded)
#pragma unroll
      for (int j = 0; j < D; ++j) {   // the box's centre; 0 when the box is not finite
        const float c = 0.5f * (lo[j] + hi[j]);
        o[j] = c - c == 0.0f ? c : 0.0f;
      }
    const float us = !ORIGIN || expanded ? 1.0f : sqrtf(gl2e);
    u64 U[P][D], S[P], G[P][D];
#pragma unroll
    for (int i = 0; i < P; ++i) {
#pragma unroll
      for (int j = 0; j < D; ++j) {
        U[i][j] = ORIGIN ? pk(us * (x[2 * i][j] - o[j]), us * (x[2 * i + 1][j] - o[j]))
                         : pk(x[2 * i][j] - o[j], x[2 * i + 1][j] - o[j]);
        G[i][j] = 0ull;
      }
      S[i] = 0ull;
    }
    // to the direct form's moments: sum w phi (x - mu) = u S - G'
    auto from_origin = [&]() {
      if (!ORIGIN || expanded) return;
      const u64 m1 = pk(-1.0f, -1.0f);
#pragma unroll
      for (int i = 0; i < P; ++i)
#pragma unroll
        for (int j = 0; j < D; ++j)
          G[i][j] = fma2(pk(x[2 * i][j] - o[j], x[2 * i + 1][j] - o[j]), S[i], mul2(G[i][j], m1));
    };
    if constexpr (L == W) {
      for (int g0 = 0; g0 < a.ngroups; g0 += kNearBatch) {
        if (g0 > 0) __syncthreads();   // every warp has walked the batch before
        const int n = near_tile<D, W, K>(a.box, a.ngroups, g0, a.M, x, act, lo, hi, expanded, gl2e, kNearSums, ns, warp,
                                         lane);
        near_sweep<D, P, ORIGIN>(a.tab, a.M, g0, NearWalk(ns, n, warp, W), expanded, o, gl2e, wraw, wbuf, lane, U, S, G);
      }
      from_origin();
      tile_finish_step<D, W, K, TRACE>(a, t, p0, act, x, o, expanded, S, G, red, warp, lane);
    } else {
      float4* buf = leaves + (CS > 1 ? (t & 1) * (L / CS) * kTile : 0);
      for (int g0 = 0; g0 < a.ngroups; g0 += kNearBatch) {
        if (g0 > 0) __syncthreads();
        const int n = near_tile<D, W, K>(a.box, a.ngroups, g0, a.M, x, act, lo, hi, expanded, gl2e, kNearSums, ns, warp,
                                         lane);
        for (int i = 0; i < L / WT; ++i) {
          near_sweep<D, P, ORIGIN>(a.tab, a.M, g0, NearWalk(ns, n, i * WT + crank * W + warp, L), expanded, o, gl2e,
                                   wraw, wbuf, lane, U, S, G);
          from_origin();
          float4* leaf = buf + (i * W + warp) * kTile;
          if (g0 == 0) tile_put_sums<D, K>(S, G, leaf, lane); else tile_add_sums<D, K>(S, G, leaf, lane);
#pragma unroll
          for (int q = 0; q < P; ++q) {
            S[q] = 0ull;
#pragma unroll
            for (int j = 0; j < D; ++j) G[q][j] = 0ull;
          }
        }
      }
      // leaf l is slot (l / WT) W + (l % WT) % W of the block of rank (l % WT) / W
      if (CS > 1) cluster_barrier(); else __syncthreads();
      // warp w updates samples 32 w + lane (a quarter of the tile, so that a
      // cluster's blocks read each other's leaves once) and shares them
      static_assert(L == W || W == K, "a warp per 32 samples");
      float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
      for (int l = 0; l < L; ++l) {
        const float4* src = buf + ((l / WT) * W + (l % WT) % W) * kTile + warp * 32 + lane;
        const float4 v = CS > 1 ? cluster_load4(cluster_addr(src, (l % WT) / W)) : *src;
        if (l == 0) acc = v; else add4(acc, v);
      }
      float xo[1][D];
      bool ao[1];
      ao[0] = p0 + warp * 32 + lane < p_end;
#pragma unroll
      for (int j = 0; j < D; ++j) xo[0][j] = x[0][j];
#pragma unroll
      for (int k = 1; k < K; ++k)
#pragma unroll
        for (int j = 0; j < D; ++j) xo[0][j] = warp == k ? x[k][j] : xo[0][j];
      tile_update<D, 1, TRACE>(a, t, p0 + warp * 32, ao, xo, o, expanded, acc, 0, crank == 0, lane);
      if (crank == 0) tile_checkpoint<D, 1>(a, t, p0 + warp * 32, ao, xo, lane);
#pragma unroll
      for (int j = 0; j < D; ++j) xs[j * kTile + warp * 32 + lane] = xo[0][j];
      __syncthreads();   // the new samples are shared, the leaves read
#pragma unroll
      for (int k = 0; k < K; ++k)
#pragma unroll
        for (int j = 0; j < D; ++j) x[k][j] = xs[j * kTile + k * 32 + lane];
    }
  }
  if (CS > 1) cluster_barrier();      // no block leaves while another may read its leaves
  tile_store<D, K, TRACE>(a, p0, act, x, writer ? 0 : 1, lane);
}

}  // namespace pdmp
