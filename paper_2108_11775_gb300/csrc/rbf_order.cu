// The order in which the sorted-tile kernels (RBF, d = 2, 3) walk a field's
// centres, and the samples' order for launches of few samples.
//
// Why the centres are ordered.  A feature w phi(x) = sign(w) 2^(lw - g' |x -
// mu|^2) is exactly zero in the kernels' arithmetic once its exponent is below
// -126: ex2.approx.ftz flushes it.  With gamma = 8 that is 3.3 units away, so
// on the fitted field of [0,10]^2 about 70 % of the features of a sample are
// such zeros (20 to 80 % on the other workloads).  With centres in Hilbert
// order and a bounding box for every 32 of them, a tile finds out from 512
// boxes (M = 16,384) which groups hold only zeros for all its samples and
// does not visit those; every other group is summed as before.  What is left
// out are additions of zero, so no result changes but by the order of its
// sums (the centres' order).  Measured: the morph of 2^20 samples (M = 16,384,
// T = 50, 2-D) 179.1 -> 59.0 ms, the log-density of 2^16 samples 37.6 -> 10.3
// ms, 48 environments 61.8 -> 42.2 ms.  The order itself takes 11 us for up to
// 4096 centres and 19 us for 16,384.
#include "kernels.cuh"
#include "order.cuh"

namespace pdmp {

// Clusters [0, chunks): one chunk of centres each.  Cluster `chunks` (if
// launched): the samples' order, for N <= kOrderChunk.
template <int D>
__global__ void __cluster_dims__(kOrderBlocks, 1, 1) __launch_bounds__(kOrderThreads)
    k_rbf_order(const float* __restrict__ centres, const float* __restrict__ w, int64_t M, int chunks,
                float4* __restrict__ tab, float4* __restrict__ box, int32_t* __restrict__ cperm, int cbits,
                const float* __restrict__ x, int N, int xbits, int32_t* __restrict__ perm) {
  __shared__ OrderSmem s;
  const int cluster = (int)(blockIdx.x / kOrderBlocks), crank = (int)(blockIdx.x % kOrderBlocks);
  if (cluster < chunks) {
    const int64_t m0 = (int64_t)cluster * kOrderChunk;
    const int n = (int)min64(kOrderChunk, M - m0);
    const int share = cluster_order<D>(centres + m0 * D, n, cbits, s, crank);
    order_table<D>(centres + m0 * D, w + m0, n, s, crank * share, share, tab + m0 * (D == 2 ? 1 : 2),
                   box + m0 / kGroup * kGroupBox, cperm + m0, m0);
  } else {
    const int share = cluster_order<D>(x, N, xbits, s, crank);
    for (int i = threadIdx.x; i < share && crank * share + i < N; i += kOrderThreads)
      perm[crank * share + i] = (int32_t)(s.items[i] & (kOrderChunk - 1));
  }
}

static size_t al256(size_t b) { return (b + 255) & ~size_t(255); }

size_t rbf_order_workspace(int d, int64_t M, int64_t N) {
  return al256((size_t)M * 16 * (d == 2 ? 1 : 2)) + al256((size_t)group_count(M) * kGroupBox * sizeof(float4)) +
         al256(sizeof(int32_t) * (size_t)M) + sort_workspace(d, N);
}

template <int D>
static cudaError_t launch_order(const float* centres, const float* w, int64_t M, const float* x, int64_t N,
                                RbfOrder& o, const SortWs& sw, cudaStream_t st) {
  const bool small = N <= kOrderChunk;
  const int chunks = (int)((M + kOrderChunk - 1) / kOrderChunk);
  cudaError_t e;
  k_rbf_order<D><<<(unsigned)(chunks + (small ? 1 : 0)) * kOrderBlocks, kOrderThreads, 0, st>>>(
      centres, w, M, chunks, o.tab, o.box, o.cperm, sort_bits(D, M < kOrderChunk ? M : kOrderChunk), x,
      small ? (int)N : 0, sw.bits, sw.perm);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return small ? cudaSuccess : spatial_sort(D, x, N, sw, st);
}

cudaError_t rbf_order(int d, const float* centres, const float* w, int64_t M, const float* x, int64_t N, void* ws,
                      RbfOrder* out, cudaStream_t st) {
  char* p = (char*)ws;
  auto take = [&](size_t b) { char* q = p; p += al256(b); return q; };
  out->tab = (float4*)take((size_t)M * 16 * (d == 2 ? 1 : 2));
  out->box = (float4*)take((size_t)group_count(M) * kGroupBox * sizeof(float4));
  out->cperm = (int32_t*)take(sizeof(int32_t) * (size_t)M);
  out->ngroups = group_count(M);
  const SortWs sw = sort_layout(p, d, N);
  out->perm = sw.perm;
  return d == 2 ? launch_order<2>(centres, w, M, x, N, *out, sw, st) : launch_order<3>(centres, w, M, x, N, *out, sw, st);
}

}  // namespace pdmp
