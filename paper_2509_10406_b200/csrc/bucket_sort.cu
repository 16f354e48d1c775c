// Stable (cluster, block) bucketing of tokens (Section "Exact retrieval": keys and values are bucketed by
// (cluster, block)): a counting sort in one launch.
#include <cooperative_groups.h>
#include "common.cuh"

namespace cg = cooperative_groups;

namespace muse {

// One problem = one thread-block cluster of up to 8 CTAs; a CTA owns a contiguous stretch of tokens that lies inside
// one spatial block (S <= 8: q = 8 / S CTAs share a block) or covers whole blocks (S > 8).  Every warp counts its own
// sub-stretch into a private histogram over the C clusters, the CTAs read each other's totals through distributed
// shared memory, and the warps then place their tokens in order, so equal keys keep ascending positions without the
// warps taking turns.  Sorting by cluster alone is enough for both orders: a query sort (block-major) is an independent
// sort of every block, and in a key sort (cluster-major) a cluster's ascending tokens already have their blocks in order.
//
// Bound by latency (three passes over a few thousand tokens per CTA and two cluster barriers).  Measured against the
// three-kernel version it replaces (a histogram, a scan over C * S * chunks counters, and a scatter in which the warps
// took turns), both sides of a clustering iteration: 8192 tokens x 16 heads 90 -> 13 us, 65536 tokens x 4 heads 145 -> 25 us.
constexpr int kSortMaxCluster = 8;

struct SortArgs { SortSide s[2]; int N, S, Bs, q; int32_t* clear; FarDefaults none; };

__global__ void __launch_bounds__(512)
k_bucket_sort(const __grid_constant__ SortArgs g) {
  extern __shared__ int32_t ssm[];
  __shared__ int32_t wsum[16];
  cg::cluster_group cluster = cg::this_cluster();
  const int CL = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int nt = blockDim.x, W = nt >> 5, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int prob = blockIdx.x / CL;
  const bool second = prob >= g.s[0].problems;
  const SortSide sd = g.s[second ? 1 : 0];
  if (second) prob -= g.s[0].problems;
  const int C = sd.C, S = g.S, N = g.N;
  int32_t* tot = ssm;                      // [C] this CTA's tokens per cluster (read by the other CTAs)
  int32_t* start = tot + C;                // [C] position of this CTA's first token of every cluster
  int32_t* hist = start + C;               // [W][C]
  pdl_wait();
  pdl_trigger();
  if (g.clear != nullptr && blockIdx.x == 0 && tid < kStatusWords) g.clear[tid] = 0;
  if (g.none.lse != nullptr && !second) {                  // (stores that nothing here waits for)
    const int step = CL * nt, nm = g.Bs * g.none.m;
    for (int e = rank * nt + tid; e < g.Bs; e += step) g.none.lse[(size_t)prob * N + e] = -INFINITY;
    for (int e = rank * nt + tid; e < nm; e += step) g.none.sel[(size_t)prob * N * g.none.m + e] = -1;
  }
  const int32_t* a = sd.assign + (size_t)prob * N;
  int32_t* pm = sd.perm + (size_t)prob * N;
  int32_t* off = sd.off + (size_t)prob * ((size_t)C * S + 1);
  // S <= 8: this CTA's part of its block; S > 8: rounds of whole blocks (queries: each block is a sort of its own)
  const int bpc = g.q > 0 ? 1 : (S + CL - 1) / CL;                                        // blocks per CTA
  const int b0 = g.q > 0 ? rank / g.q : rank * bpc;
  const int part = g.q > 0 ? rank % g.q : 0;
  const int rounds = sd.kind == 0 ? bpc : 1;
  for (int r = 0; r < rounds; ++r) {
    const int b = b0 + r;
    int t0, t1;
    if (g.q > 0) {
      const int per = (g.Bs + g.q - 1) / g.q;
      t0 = b * g.Bs + min(g.Bs, part * per);
      t1 = b * g.Bs + min(g.Bs, (part + 1) * per);
    } else if (sd.kind == 0) {
      t0 = min(b, S) * g.Bs; t1 = min(b + 1, S) * g.Bs;
    } else {
      t0 = min(b0, S) * g.Bs; t1 = min(b0 + bpc, S) * g.Bs;
    }
    const int wl = ((t1 - t0 + W - 1) / W + 31) & ~31;                                    // tokens per warp
    const int w0 = min(t1, t0 + warp * wl), w1 = min(t1, w0 + wl);
    int32_t* h = hist + (size_t)warp * C;
    for (int k = tid; k < W * C; k += nt) hist[k] = 0;
    __syncthreads();
    for (int t = w0 + lane; t < w1; t += 128) {
      int v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = t + 32 * u < w1 ? a[t + 32 * u] : -1;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (t + 32 * u < w1) atomicAdd(&h[min(max(v[u], 0), C - 1)], 1);                  // (an assignment outside [0, C) is pinned)
    }
    __syncthreads();
    for (int k = tid; k < C; k += nt) {                                                   // exclusive prefix over the warps
      int run = 0;
      for (int w = 0; w < W; ++w) { const int x = hist[(size_t)w * C + k]; hist[(size_t)w * C + k] = run; run += x; }
      tot[k] = run;
    }
    if (sd.kind == 1 || g.q > 1) cluster.sync(); else __syncthreads();
    // clusters' totals over the CTAs that sort together, this CTA's share in front, and the scan over the clusters
    const int r0 = sd.kind == 0 ? rank - part : 0, r1 = sd.kind == 0 ? (g.q > 0 ? r0 + g.q : rank + 1) : CL;
    const int rr0 = sd.kind == 0 && g.q == 0 ? rank : r0;
    const int per = (C + nt - 1) / nt, k0 = min(C, tid * per), k1 = min(C, k0 + per);
    int mine = 0;
    for (int k = k0; k < k1; ++k) {
      int before = 0, all = 0;
      for (int o = rr0; o < r1; ++o) {
        const int x = *cluster.map_shared_rank(&tot[k], o);
        if (o < rank) before += x;
        all += x;
      }
      start[k] = mine + before;
      mine += all;
    }
    int inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int x = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += x; }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    int base = inc - mine + (sd.kind == 0 ? min(b, S) * g.Bs : 0);
    for (int w = 0; w < warp; ++w) base += wsum[w];
    for (int k = k0; k < k1; ++k) {
      const int p = base + start[k];
      start[k] = p;
      if (sd.kind == 0) { if (part == 0 && b < S) off[(size_t)b * C + k] = p; }
      else if (g.q > 0) { if (part == 0) off[(size_t)k * S + b] = p; }
      else if (rank == 0) off[(size_t)k * S] = p;
    }
    if (tid == 0 && rank == 0 && r == 0) off[(size_t)C * S] = N;
    __syncthreads();
    // every warp places its tokens in order
    for (int tb = w0; tb < w1; tb += 128) {
      int v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = tb + 32 * u + lane < w1 ? min(max(a[tb + 32 * u + lane], 0), C - 1) : -1 - lane;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (tb + 32 * u >= w1) break;
        const int key = v[u];
        const unsigned peers = __match_any_sync(0xffffffffu, key);
        const int rk = __popc(peers & ((1u << lane) - 1u));
        const int at = key >= 0 ? h[key] : 0;
        __syncwarp();
        if (key >= 0) {
          if (rk == 0) h[key] = at + __popc(peers);
          const int p = start[key] + at + rk;
          if (MUSE_IN_RANGE(p, N)) pm[p] = tb + 32 * u + lane;
        }
        __syncwarp();
      }
    }
    __syncthreads();
  }
  if (sd.kind == 1 && g.q == 0) __threadfence();
  cluster.sync();                          // no CTA leaves (or reuses its totals) while another may still read them
  if (sd.kind == 1 && g.q == 0) {
    // more than 8 blocks: a cluster's tokens ascend, so its blocks' first positions are found by bisection
    for (int e = rank * nt + tid; e < C * (S - 1); e += CL * nt) {
      const int j = e / (S - 1), b = e % (S - 1) + 1;
      int lo = __ldcg(&off[(size_t)j * S]), hi = j + 1 < C ? __ldcg(&off[(size_t)(j + 1) * S]) : N;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (__ldcg(&pm[mid]) < b * g.Bs) lo = mid + 1; else hi = mid;
      }
      off[(size_t)j * S + b] = lo;
    }
  }
}

int bucket_sort(const SortSide* sides, int nsides, int N, int S, int Bs, cudaStream_t st, int32_t* clear, const FarDefaults* none) {
  SortArgs g = {};
  int total = 0, C = 0;
  for (int k = 0; k < nsides; ++k) { g.s[k] = sides[k]; total += sides[k].problems; C = C > sides[k].C ? C : sides[k].C; }
  g.N = N; g.S = S; g.Bs = Bs; g.clear = clear;
  if (none != nullptr) g.none = *none;
  g.q = S <= kSortMaxCluster ? kSortMaxCluster / S : 0;
  const int cl = g.q > 0 ? S * g.q : kSortMaxCluster;
  const int warps = C <= 2048 ? 16 : 8;                                    // private histograms of at most 128 KB
  prof_mark("k_bucket_sort", st);
  return launch_pdl_cluster(k_bucket_sort, dim3(total * cl), warps * 32, (size_t)(2 + warps) * C * sizeof(int32_t), cl, st, g);
}

}  // namespace muse
