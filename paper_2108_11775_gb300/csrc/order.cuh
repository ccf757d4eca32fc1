// Spatial order of a field's centres and the boxes of its groups of centres
// (see rbf_order.cu), with which a sample tile leaves out the groups whose
// every feature is exactly zero on it.
#pragma once
#include "sort.cuh"

namespace pdmp {

// Centres are ordered in chunks of kOrderChunk (a cluster of kOrderBlocks
// blocks each), and the sweeps take them in groups of kGroup consecutive ones:
// one warp stage.
constexpr int kOrderChunk = 16384;
constexpr int kOrderBlocks = 8;      // blocks per cluster
constexpr int kOrderThreads = 512;
constexpr int kOrderWarps = kOrderThreads / 32;
constexpr int kOrderShare = kOrderChunk / kOrderBlocks;   // items per block at most
constexpr int kGroup = 32;
constexpr int kGroupBox = 3;         // float4s per group: its bounding box, its strongest centre and log2|w|
constexpr int kDigits = 64;          // radix of the sort (keys of two digits)
constexpr int kCountRow = kOrderWarps + 1;   // rows padded: a warp's lanes hit distinct banks
static_assert(kDigits * kOrderBlocks == kOrderThreads, "a thread per digit and block");

struct OrderSmem {
  uint32_t items[kOrderShare];       // sorted: key << 14 | index within the chunk (this block's positions)
  uint32_t other[kOrderShare];       // the items between the two passes
  uint16_t rank[kOrderShare];
  uint32_t count[kDigits * kCountRow];   // [digit][warp]
  uint32_t total[kDigits];           // this block's items of each digit
  uint32_t base[kDigits];            // where they go
  uint32_t scan[33];
  float red[6 * kOrderWarps];
  float box[6];
  uint32_t curve[48];                // the 3-D curve's table
};

// shared::cluster address of a shared-memory object in the cluster's block `rank`
__device__ __forceinline__ uint32_t cluster_addr(const void* p, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ uint32_t cluster_load(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ float4 cluster_load4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}
__device__ __forceinline__ void cluster_store(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
// every thread of the cluster; orders shared memory accesses across it
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_barrier() {
  cluster_arrive();
  cluster_wait();
}

// hilbert_key as an automaton, a lookup per level instead of the reflections
// and exchanges of all lower bits: for state s and the level's cell bits q (c_0
// most significant) the table gives the index digit and the next state.  Both
// tables were generated from hilbert_key and reproduce it for every input.
// 2-D: 4 states, 4 bits an entry (digit | state << 2), entry 4 s + q.
constexpr uint64_t kCurve2 = 0x8d7ec39a65f02b14ull;
// 3-D: 24 states, a byte an entry (digit | state << 3), entry 8 s + q.
static __device__ const uint32_t kCurve3[48] = {
    0x021b1108u, 0x05342e27u, 0x56494738u, 0x0d0a145bu, 0x6e670130u, 0x150c1273u, 0x1a1d817eu, 0x038c504fu,
    0x22252b94u, 0x514e807fu, 0x2a232d9cu, 0x69a0061fu, 0x048b5748u, 0x35324639u, 0x4c6fab00u, 0x3d663a31u,
    0xb8538fb4u, 0x61423645u, 0x4a097b10u, 0x4d263c2fu, 0x0e555f84u, 0x21529043u, 0x60b9378eu, 0x0b5a745du,
    0xb0af6bbcu, 0x413e6265u, 0x16776da4u, 0x29986a63u, 0x403fb1aeu, 0x135c7275u, 0x7aa17d1eu, 0x4b68ac07u,
    0xa6851982u, 0xbf5488b3u, 0x1c8d0f5eu, 0x338a2091u, 0x24959b92u, 0xa7be1889u, 0x2c939d9au, 0x8778b6a9u,
    0x8679a5a2u, 0xb7a86cbbu, 0x7c17ad76u, 0x3b28aa99u, 0x588371b2u, 0x97449eb5u, 0x7059a3bau, 0x9f9664bdu};

template <int D>
__device__ __forceinline__ uint32_t curve_key(const uint32_t (&c)[D], int bits, const uint32_t* curve) {
  uint32_t key = 0, s = 0;
  for (int b = bits - 1; b >= 0; --b) {
    uint32_t q = 0;
#pragma unroll
    for (int j = 0; j < D; ++j) q = q << 1 | (c[j] >> b & 1u);
    if (D == 2) {
      const uint32_t e = (uint32_t)(kCurve2 >> ((s << 2 | q) << 2));
      key = key << 2 | (e & 3u);
      s = e >> 2 & 3u;
    } else {
      const uint32_t e = reinterpret_cast<const uint8_t*>(curve)[s << 3 | q];
      key = key << 3 | (e & 7u);
      s = e >> 3;
    }
  }
  return key;
}

// Exclusive prefix sum over the block's threads (blockDim.x a multiple of 32,
// at most 1024) of v; total receives the sum.  sh: 33 words.
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* sh, uint32_t& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) sh[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0u;
    uint32_t wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t t = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += t;
    }
    sh[lane] = wi - w;
    if (lane == 31) sh[32] = wi;
  }
  __syncthreads();
  uint32_t r = inc - v + sh[warp];
  total = sh[32];
  __syncthreads();
  return r;
}

// A cluster of kOrderBlocks blocks of kOrderThreads orders n <= kOrderChunk
// points by the Hilbert index of their grid cell (2^bits cells an axis over the
// points' bounding box, 2^(D bits) <= 4096 cells), points of a cell by index: a
// stable radix sort of two 6-bit digits, so the order depends on the points
// alone.  Block `crank` holds a share of the input and ends up with the sorted
// positions [crank * share, (crank + 1) * share) in s.items (index = low 14
// bits); returns share.  A warp's items are consecutive, its lanes' ranks come
// from ballots on their digits, no atomics are used; the blocks exchange
// bounding boxes, digit totals and the items through each other's shared
// memory.  One block alone took 62 us for 16,384 points (some 370 instructions
// a point, issued by one SM).
template <int D>
__device__ int cluster_order(const float* __restrict__ pts, int n, int bits, OrderSmem& s, int crank) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (D == 3 && threadIdx.x < 48) s.curve[threadIdx.x] = kCurve3[threadIdx.x];
  // rounds of kOrderThreads items per block: 1, 2 or 4
  const int lg = n <= kOrderBlocks * kOrderThreads ? 0 : (n <= 2 * kOrderBlocks * kOrderThreads ? 1 : 2);
  const int rounds = 1 << lg, share = kOrderThreads << lg, lgshare = 9 + lg;
  static_assert(kOrderThreads == 512, "lgshare");
  const int first = warp * 32 * rounds + lane, i0 = crank * share;
  float lo[D], hi[D];
#pragma unroll
  for (int j = 0; j < D; ++j) { lo[j] = INFINITY; hi[j] = -INFINITY; }
#pragma unroll 4
  for (int r = 0; r < rounds; ++r) {
    const int i = i0 + first + 32 * r;
    if (i < n)
#pragma unroll
      for (int j = 0; j < D; ++j) {
        const float v = pts[(size_t)i * D + j];
        if (v == v) { lo[j] = fminf(lo[j], v); hi[j] = fmaxf(hi[j], v); }
      }
  }
#pragma unroll
  for (int j = 0; j < D; ++j) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      lo[j] = fminf(lo[j], __shfl_xor_sync(0xffffffffu, lo[j], o));
      hi[j] = fmaxf(hi[j], __shfl_xor_sync(0xffffffffu, hi[j], o));
    }
    if (lane == 0) {
      s.red[j * kOrderWarps + warp] = lo[j];
      s.red[(D + j) * kOrderWarps + warp] = hi[j];
    }
  }
  __syncthreads();
  if (threadIdx.x < 2 * D) {
    float v = s.red[threadIdx.x * kOrderWarps];
    for (int w = 1; w < kOrderWarps; ++w) {
      const float u = s.red[threadIdx.x * kOrderWarps + w];
      v = threadIdx.x < D ? fminf(v, u) : fmaxf(v, u);
    }
    s.box[threadIdx.x] = v;
  }
  cluster_barrier();
#pragma unroll
  for (int j = 0; j < D; ++j) {
    // lanes 0 .. 7 read the blocks' boxes
    lo[j] = __uint_as_float(cluster_load(cluster_addr(&s.box[j], lane & (kOrderBlocks - 1))));
    hi[j] = __uint_as_float(cluster_load(cluster_addr(&s.box[D + j], lane & (kOrderBlocks - 1))));
#pragma unroll
    for (int o = kOrderBlocks / 2; o > 0; o >>= 1) {
      lo[j] = fminf(lo[j], __shfl_xor_sync(0xffffffffu, lo[j], o));
      hi[j] = fmaxf(hi[j], __shfl_xor_sync(0xffffffffu, hi[j], o));
    }
  }
  const float cells = (float)(1u << bits);
  float scale[D];
#pragma unroll
  for (int j = 0; j < D; ++j) scale[j] = cell_scale(lo[j], hi[j], cells);
#pragma unroll 4
  for (int r = 0; r < rounds; ++r) {
    const int i = i0 + first + 32 * r;
    uint32_t key = 0xfffu;   // past the end: after every point of the last cell
    if (i < n) {
      uint32_t c[D];
#pragma unroll
      for (int j = 0; j < D; ++j) c[j] = cell_at(pts[(size_t)i * D + j], lo[j], scale[j], cells);
      key = curve_key<D>(c, bits, s.curve);
    }
    s.items[first + 32 * r] = key << 14 | (uint32_t)i;
  }
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    const uint32_t* src = pass == 0 ? s.items : s.other;
    const uint32_t* dst = pass == 0 ? s.other : s.items;
    const int shift = 14 + 6 * pass;
    for (int i = threadIdx.x; i < kDigits * kCountRow; i += kOrderThreads) s.count[i] = 0u;
    __syncthreads();
#pragma unroll 2
    for (int r = 0; r < rounds; ++r) {
      const uint32_t dgt = src[first + 32 * r] >> shift & (kDigits - 1);
      uint32_t same = 0xffffffffu;       // the lanes with this digit (six ballots: the match instruction is slower)
#pragma unroll
      for (int b = 0; b < 6; ++b) {
        const uint32_t set = __ballot_sync(0xffffffffu, dgt >> b & 1u);
        same &= dgt >> b & 1u ? set : ~set;
      }
      const uint32_t before = s.count[dgt * kCountRow + warp];
      s.rank[first + 32 * r] = (uint16_t)(before + __popc(same & ((1u << lane) - 1u)));
      __syncwarp();
      if (lane == __ffs(same) - 1) s.count[dgt * kCountRow + warp] = before + __popc(same);
      __syncwarp();
    }
    __syncthreads();
    if (threadIdx.x < kDigits) {         // within the digit: the warps before
      uint32_t acc = 0;
      for (int w = 0; w < kOrderWarps; ++w) {
        const uint32_t c = s.count[threadIdx.x * kCountRow + w];
        s.count[threadIdx.x * kCountRow + w] = acc;
        acc += c;
      }
      s.total[threadIdx.x] = acc;
    }
    cluster_barrier();
    // thread (digit, block): the items of smaller digits, and of this digit in the blocks before
    const int blk = threadIdx.x & (kOrderBlocks - 1), dig = threadIdx.x / kOrderBlocks;
    uint32_t all;
    const uint32_t ex = block_exclusive_scan(cluster_load(cluster_addr(&s.total[dig], blk)), s.scan, all);
    if (blk == crank) s.base[dig] = ex;
    __syncthreads();
#pragma unroll 2
    for (int r = 0; r < rounds; ++r) {
      const uint32_t it = src[first + 32 * r], dgt = it >> shift & (kDigits - 1);
      const uint32_t pos = s.base[dgt] + s.count[dgt * kCountRow + warp] + s.rank[first + 32 * r];
      cluster_store(cluster_addr(&dst[pos & (share - 1)], (int)(pos >> lgshare)), it);
    }
    cluster_barrier();
  }
  return share;
}

// Table entries and group boxes of the sorted positions [p0, p0 + share) that
// this block holds of a chunk of n centres: entry i of the chunk is {mu_0 ..
// mu_{D-1}, lw = log2|w|, sg = sign(w)} of the centre there; perm (may be
// NULL) receives base + its index in the chunk.  Box of a group: {lo_0 ..,
// lw_max in .w}, {hi_0 ..}, {mu_0 .., lw in .w} of its centre of largest |w|; a
// centre or weight that is not finite makes its group's box everything, so
// that no tile leaves the group out.
template <int D>
__device__ void order_table(const float* __restrict__ centres, const float* __restrict__ w, int n, const OrderSmem& s,
                            int p0, int share, float4* __restrict__ tab, float4* __restrict__ box,
                            int32_t* __restrict__ perm, int64_t base) {
  const int lane = threadIdx.x & 31, warps = kOrderWarps;
  const int end = n < p0 + share ? n : p0 + share;
  constexpr int U = 4;   // groups in flight per warp: the gathers' latency is what this takes
  for (int g0 = p0 / kGroup + (threadIdx.x >> 5); g0 * kGroup < end; g0 += U * warps) {
    float mu[U][D], wm[U];
    int m[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = (g0 + u * warps) * kGroup + lane;
      m[u] = i < end ? (int)(s.items[i - p0] & (kOrderChunk - 1)) : -1;
      wm[u] = m[u] >= 0 ? w[m[u]] : 0.0f;
#pragma unroll
      for (int j = 0; j < D; ++j) mu[u][j] = m[u] >= 0 ? centres[(size_t)m[u] * D + j] : 0.0f;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int g = g0 + u * warps, i = g * kGroup + lane;
      if (g * kGroup >= end) break;
      float lo[D], hi[D], lmax = -INFINITY;
      bool odd = false;
#pragma unroll
      for (int j = 0; j < D; ++j) { lo[j] = INFINITY; hi[j] = -INFINITY; }
      if (i < end) {
        const float lw = wm[u] != 0.0f ? log2f(fabsf(wm[u])) : -INFINITY;
        const float sg = wm[u] > 0.0f ? 1.0f : (wm[u] < 0.0f ? -1.0f : 0.0f);
#pragma unroll
        for (int j = 0; j < D; ++j) {
          lo[j] = hi[j] = mu[u][j];
          odd = odd || !(fabsf(mu[u][j]) < INFINITY);
        }
        odd = odd || !(fabsf(wm[u]) < INFINITY);
        lmax = lw;
        if (D == 2) {
          tab[i] = make_float4(mu[u][0], mu[u][1], lw, sg);
        } else {
          tab[2 * i] = make_float4(mu[u][0], mu[u][1], mu[u][D - 1], lw);
          tab[2 * i + 1] = make_float4(sg, 0.0f, 0.0f, 0.0f);
        }
        if (perm) perm[i] = (int32_t)(base + m[u]);
      }
      odd = __any_sync(0xffffffffu, odd);
      const float lw0 = lmax;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        lmax = fmaxf(lmax, __shfl_xor_sync(0xffffffffu, lmax, o));
#pragma unroll
        for (int j = 0; j < D; ++j) {
          lo[j] = fminf(lo[j], __shfl_xor_sync(0xffffffffu, lo[j], o));
          hi[j] = fmaxf(hi[j], __shfl_xor_sync(0xffffffffu, hi[j], o));
        }
      }
      const int top = __ffs(__ballot_sync(0xffffffffu, i < end && lw0 == lmax)) - 1;
      float mt[D];
#pragma unroll
      for (int j = 0; j < D; ++j) mt[j] = __shfl_sync(0xffffffffu, mu[u][j], top < 0 ? 0 : top);
      const float lt = odd ? -INFINITY : lmax;
      if (lane == 0) {
        if (odd) {
          lmax = INFINITY;
#pragma unroll
          for (int j = 0; j < D; ++j) { lo[j] = -INFINITY; hi[j] = INFINITY; }
        }
        box[kGroupBox * g] = make_float4(lo[0], lo[1], D == 3 ? lo[D - 1] : 0.0f, lmax);
        box[kGroupBox * g + 1] = make_float4(hi[0], hi[1], D == 3 ? hi[D - 1] : 0.0f, 0.0f);
        box[kGroupBox * g + 2] = make_float4(mt[0], mt[1], D == 3 ? mt[D - 1] : 0.0f, lt);
      }
    }
  }
}

// what a sorted-tile launch works on: the ordered centre table with its
// groups' boxes, and the samples' order
struct RbfOrder {
  float4* tab;
  float4* box;
  int32_t* cperm;    // table position -> centre
  int32_t* perm;     // sorted position -> sample
  int ngroups;
};

__host__ __device__ __forceinline__ int group_count(int64_t M) { return (int)((M + kGroup - 1) / kGroup); }
size_t rbf_order_workspace(int d, int64_t M, int64_t N);
// centres (RBF, d = 2, 3) and samples into ws (rbf_order_workspace bytes)
cudaError_t rbf_order(int d, const float* centres, const float* w, int64_t M, const float* x, int64_t N, void* ws,
                      RbfOrder* out, cudaStream_t st);

}  // namespace pdmp
