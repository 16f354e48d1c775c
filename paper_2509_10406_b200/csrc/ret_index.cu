// Inverse index for retrieval (Section "Exact Retrieval and Local Attention"): for every (key cluster, plane) the list of
// (query, slot) pairs that retrieve it.  Group key = cluster * SB + plane, so that the pairs of one cluster over all planes
// form one run, ordered by plane.  With spatial block selection (bsel, k2 > 0) a pair is (query, slot, chosen block e), its
// group the BUCKET (cluster, chosen block) and its id (query * m + slot) * k2 + e.
//
// One launch: a head is one thread-block cluster, a CTA owns a stretch of its tokens.  Every CTA counts its pairs by key in
// shared memory; the CTAs split the keys, read each other's counts through distributed shared memory and write back where
// in the list each CTA's pairs of a key start; then every CTA goes over its pairs again and places them.  The first CTA also lists
// the shares in which the tensor-core kernels take the groups.
//
// Bound by the scattered 4-byte stores of the last pass (a store per lane) and shared-memory atomics.  32 heads of 64k tokens,
// 8 slots, 128 clusters, 8 blocks: 126 us (161 with two divisions a pair for its plane); a memset, a counting kernel, a scan and a
// placing kernel that combined equal keys of a warp into one global atomic took 1480 us.  4 heads of 128k, 32 slots, 2048 clusters
// 348 -> 275; 4 heads of 64k, 32 slots, 1024 clusters 184 -> 148; 16 heads of 8k, whose few pairs a CTA keeps between the passes,
// 37 -> 31.
#include <cooperative_groups.h>
#include "common.cuh"

namespace cg = cooperative_groups;

namespace muse {

constexpr int kRiThreads = 1024, kRiMaxCluster = 16, kRiMinPairs = 2048, kRiKept = 8;   // kept: pairs of a thread that stay in registers between the passes

struct RiArgs { const int32_t *sel, *bsel, *off_k; RetIndex ri; int nkeys; };

__global__ void __launch_bounds__(kRiThreads)
k_ret_index(Dims d, const __grid_constant__ RiArgs g) {
  extern __shared__ int32_t hist[];                        // [nkeys] counts of this CTA's pairs; then where the next pair of a key goes
  __shared__ int32_t wsum[32], share_s[kRiMaxCluster];
  cg::cluster_group cluster = cg::this_cluster();
  const int CL = (int)cluster.num_blocks(), rank = (int)cluster.block_rank(), pq = blockIdx.x / CL;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nkeys = g.nkeys, ke = g.bsel ? d.k2 : 1;
  const int per = (d.N + CL - 1) / CL, t0 = min(d.N, rank * per), t1 = min(d.N, t0 + per);
  for (int k = tid; k < nkeys; k += kRiThreads) hist[k] = 0;
  pdl_wait();
  pdl_trigger();
  __syncthreads();
  // the key of pair `e` (counted over the CTA's tokens and slots), or -1: entries outside [0, Ck) count as "none"
  const int n = (t1 - t0) * d.m;
  const int32_t* sel = g.sel + ((size_t)pq * d.N + t0) * d.m;
  const int32_t* bsel = g.bsel ? g.bsel + ((size_t)pq * d.N + t0) * d.m * ke : nullptr;
  // (a thread's pairs ascend, so their plane is followed from block to block: two divisions a pair were a third of the instructions)
  struct Plane { int pl; unsigned end; };                  // of the next pair, and the first pair of a later block
  const unsigned bm = (unsigned)d.Bs * d.m;
  const Plane pl0 = d.causal ? Plane{t0 / d.Bs - 1, (unsigned)(t0 / d.Bs + 1) * bm - (unsigned)t0 * d.m} : Plane{0, 0xffffffffu};
  auto key_of = [&](Plane& p, int e, int c, int x) {
    while ((unsigned)e >= p.end) { ++p.pl; p.end = p.pl + 1 < d.S - 1 ? p.end + bm : 0xffffffffu; }
    const int pl = p.pl;                                   // block 0 sees no other block
    if (c < 0 || c >= d.Ck || pl < 0) return -1;
    if (bsel == nullptr) return c * d.SB + pl;
    const int bb = bsel[(size_t)e * ke + x];
    return bb < 0 || bb > pl ? -1 : c * d.SB + bb;                             // (an earlier block than the query's block pl + 1)
  };
  constexpr int U = 4;                                     // pairs in flight per thread
  // a CTA of few pairs counts and remembers what the count said: key | place among the CTA's pairs of the key << 15
  const bool keep = ke == 1 && g.bsel == nullptr && n <= kRiKept * kRiThreads;
  uint32_t kept[kRiKept];
  Plane p = pl0;
  if (keep) {
    int c[kRiKept];
#pragma unroll
    for (int u = 0; u < kRiKept; ++u) c[u] = tid + u * kRiThreads < n ? sel[tid + u * kRiThreads] : -1;
#pragma unroll
    for (int u = 0; u < kRiKept; ++u) {
      const int key = c[u] >= 0 ? key_of(p, tid + u * kRiThreads, c[u], 0) : -1;
      kept[u] = key >= 0 ? (uint32_t)key | (uint32_t)atomicAdd(&hist[key], 1) << 15 : 0xffffffffu;
    }
  }
  for (int e0 = tid; !keep && e0 < n; e0 += U * kRiThreads) {
    int c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) c[u] = e0 + u * kRiThreads < n ? sel[e0 + u * kRiThreads] : -1;
#pragma unroll
    for (int u = 0; u < U; ++u)
      for (int x = 0; x < ke; ++x) {
        const int key = key_of(p, e0 + u * kRiThreads, c[u], x);
        if (key >= 0) atomicAdd(&hist[key], 1);
      }
  }
  cluster.sync();
  // this CTA's share of the keys: totals over the CTAs, their exclusive prefix within the share
  const int kper = (nkeys + CL - 1) / CL, ka = min(nkeys, rank * kper), kb = min(nkeys, ka + kper);
  int32_t* goff = g.ri.goff + (size_t)pq * (nkeys + 1);
  int share = 0, v[kRiMaxCluster], all = 0;                // counts of a key in every CTA
  auto counts = [&](int k) {
    all = 0;
#pragma unroll
    for (int c = 0; c < kRiMaxCluster; ++c) {
      v[c] = c < CL && k < kb ? cluster.map_shared_rank(hist, min(c, CL - 1))[k] : 0;
      all += v[c];
    }
  };
  for (int k0 = ka; k0 < kb; k0 += kRiThreads) { counts(k0 + tid); share += all; }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) share += __shfl_xor_sync(0xffffffffu, share, o);
  if (lane == 0) wsum[warp] = share;
  __syncthreads();
  if (warp == 0) {
    int v = wsum[lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane < CL) cluster.map_shared_rank(share_s, lane)[rank] = v;
  }
  cluster.sync();
  int carry = 0;                                           // pairs before this share
  for (int c = 0; c < rank; ++c) carry += share_s[c];
  for (int k0 = ka; k0 < kb; k0 += kRiThreads) {
    const int k = k0 + tid;
    if (kper > kRiThreads) counts(k);                      // (else this thread's one key is still here)
    int inc = all;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int x = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += x; }
    __syncthreads();
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    int at = carry + inc - all;
    for (int w = 0; w < 32; ++w) { const int x = wsum[w]; if (w < warp) at += x; carry += x; }
    if (k < kb) {
      goff[k] = at;
#pragma unroll
      for (int c = 0; c < kRiMaxCluster; ++c)
        if (c < CL) { cluster.map_shared_rank(hist, c)[k] = at; at += v[c]; }
    }
  }
  if (rank == CL - 1 && tid == 0) goff[nkeys] = carry;
  cluster.sync();
  if (rank == 0) {                                         // the shares of every group's pairs (this CTA has the tokens of block 0, which have no pairs)
    const int stride = g.bsel ? 1 : d.SB, G = nkeys / stride;
    RetItem* items = g.ri.items + (size_t)pq * g.ri.cap;
    const int32_t* ok = g.off_k + (size_t)(pq / d.Hq * d.Hkv + d.hm.g[pq % d.Hq]) * (d.Ck * d.S + 1);
    int carry2 = 0;
    for (int k0 = 0; k0 < G; k0 += kRiThreads) {
      const int k = k0 + tid, p0 = k < G ? __ldcg(goff + k * stride) : 0, p1 = k < G ? __ldcg(goff + (k + 1) * stride) : 0, np = p1 - p0;
      const int b0 = g.bsel ? k / d.SB * d.S + k % d.SB : k * d.S;             // the group's first bucket; it ends with that one, or with the block SB
      const int kf = k < G ? ok[b0] : 0, nk = k < G ? ok[b0 + (g.bsel ? 1 : d.SB)] - kf : 0;
      const int tiles = (np + kRetTile - 1) / kRetTile, ns = min(32767, (tiles + g.ri.share - 1) / g.ri.share);
      int inc = ns;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += v; }
      __syncthreads();
      if (lane == 31) wsum[warp] = inc;
      __syncthreads();
      int at = carry2 + inc - ns;
      for (int w = 0; w < 32; ++w) { const int v = wsum[w]; if (w < warp) at += v; carry2 += v; }
      for (int s = 0; s < ns; ++s)
        if (MUSE_IN_RANGE(at + s, g.ri.cap)) items[at + s] = RetItem{k, s | ns << 16, p0, p1, kf, nk, {0, 0}};
    }
    if (tid == 0) g.ri.nitems[pq] = carry2;
  }
  const size_t npairs = (size_t)d.N * d.m * ke;
  int32_t* pairs = g.ri.pairs + (size_t)pq * npairs;
  if (keep) {
#pragma unroll
    for (int u = 0; u < kRiKept; ++u) {
      if (kept[u] == 0xffffffffu) continue;
      const int at = hist[kept[u] & 0x7fffu] + (int)(kept[u] >> 15);
      if (MUSE_IN_RANGE(at, npairs)) pairs[at] = t0 * d.m + tid + u * kRiThreads;
    }
    return;
  }
  p = pl0;
  for (int e0 = tid; e0 < n; e0 += U * kRiThreads) {
    int c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) c[u] = e0 + u * kRiThreads < n ? sel[e0 + u * kRiThreads] : -1;
    const Plane p0 = p;
    for (int x = 0; x < ke; ++x) {
      p = p0;
      int at[U];                                           // (the places of all before the first store: the atomics overlap)
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int key = key_of(p, e0 + u * kRiThreads, c[u], x);
        at[u] = key >= 0 ? atomicAdd(&hist[key], 1) : -1;
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (at[u] >= 0 && MUSE_IN_RANGE(at[u], npairs)) pairs[at[u]] = (t0 * d.m + e0 + u * kRiThreads) * ke + x;
    }
  }
}

static size_t up64(size_t x) { return (x + 63) & ~size_t(63); }
static int item_cap(const Dims& d, int share) {
  const int groups = d.k2 > 0 ? d.Ck * d.SB : d.Ck;
  return (int)((long long)d.N * d.m * (d.k2 > 0 ? d.k2 : 1) / (kRetTile * share)) + groups;
}

size_t ret_index_elems(const Dims& d) {
  // goff [SB*Ck+1] + pairs [N*m*max(k2,1)] + items (8 each) + their number, each rounded up to 64 ints
  return up64((size_t)d.SB * d.Ck + 1) + up64((size_t)d.N * d.m * (d.k2 > 0 ? d.k2 : 1)) + up64(8 * (size_t)item_cap(d, kMinShare)) + 64;
}

int build_ret_index(const Dims& d, const int32_t* sel, const int32_t* bsel, const int32_t* off_k, int32_t* scratch, RetIndex* out, cudaStream_t st) {
  const int pq = d.B * d.Hq, nkeys = d.SB * d.Ck, mk = d.m * (bsel ? d.k2 : 1);        // nkeys <= 32768
  // Shares of 32 tiles; fewer where that would leave SMs without work (selections crowd on few clusters: one may have all of a head's
  // queries), not below 4 (a share loads its keys and adds its gradients once).
  const long long tiles = (long long)d.N * mk * pq / kRetTile, want = tiles / (8 * sm_count());
  out->share = (int)(want < kMinShare ? kMinShare : want > kMaxShare ? kMaxShare : want);
  out->cap = item_cap(d, out->share);
  out->goff = scratch;                                     // (indexed with its natural stride, nkeys + 1)
  out->pairs = out->goff + (size_t)pq * up64((size_t)nkeys + 1);
  out->items = (RetItem*)(out->pairs + (size_t)pq * up64((size_t)d.N * mk));
  out->nitems = (int32_t*)(out->items + (size_t)pq * up64(8 * (size_t)item_cap(d, kMinShare)) / 8);
  if (d.m == 0 || nkeys == 0) return MUSE_OK;
  // CTAs of a head, of 2048 pairs or more: until half the SMs have one (a large cluster pays in its exchange of counts and in scheduling:
  // 32 heads of 16k tokens, 16 slots 131 us with 8 CTAs, 87 with 4; 4 heads of 64k, 32 slots 181 us with 16, 326 with 8)
  int cl = 1;
  while (cl < kRiMaxCluster && cl * pq < sm_count() / 2 && (long long)d.N * d.m >= 2LL * cl * kRiMinPairs) cl *= 2;
  const size_t smem = (size_t)nkeys * sizeof(int32_t);
  const RiArgs g = {sel, bsel, off_k, *out, nkeys};
  // More than 8 CTAs are not promised by every device: they have to share a processor group, each with up to 128 KB of shared memory.
  if (cl > 8 && !cluster_fits(k_ret_index, kRiThreads, smem, cl)) cl = 8;
  prof_mark("k_ret_index", st);
  return launch_pdl_cluster(k_ret_index, dim3(pq * cl), kRiThreads, smem, cl, st, d, g);
}

}  // namespace muse
