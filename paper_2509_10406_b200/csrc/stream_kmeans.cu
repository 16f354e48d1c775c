// The paper's own clustering (Appendix "Clustering Details").
//
// "Centroid Computation": one pass of streaming mini-batch k-means.  The N vectors of a problem (one head,
// queries or keys) are visited in the order of the seeded shuffle, 64 at a time; a minibatch is assigned to
// the nearest current centroids t_j / c_j, then its vectors update their centroids one after the other,
// t_j <- beta t_j + x, c_j <- beta c_j + 1.  Centroid r starts as the r-th strided sample of the shuffled
// sequence with t = x, c = 1.  The pass is a chain of N / 64 dependent steps, so a problem is owned by one
// thread-block cluster (its CTAs split the centroids) and the problems run side by side; a step is a
// 64 x C x D distance product (fp32 FFMA on shared-memory tiles of 64 vectors x 64 centroids, 4 x 2 results
// per thread), an arg-min with ties to the lower index, and the update, in which one warp per touched centroid
// replays that centroid's vectors of the minibatch in stream order - exactly the sequential recurrence,
// parallel over centroids.  The next minibatch's rows are fetched while the current one is worked on.
//
// "Balanced Assignment": independently in each spatial block every vector goes to its nearest centroid
// subject to a bucket size of at most cap = ceil(factor * B / K).  Step 1 (data parallel): the nearest
// centroid of every vector (the assignment kernels of the Lloyd path), a stable (block, cluster) counting
// sort, and each vector's rank inside its bucket in position order; the first cap of a bucket keep it.
// Step 2: one CTA per (problem, block) walks the displaced vectors in position order and gives each the
// nearest centroid whose bucket still has room: a masked arg-min over one row of a distance matrix, which is written
// only for the 128-vector tiles that hold a displaced vector.  Where the cap rarely binds (the paper's regime: 128 clusters, cap 256 per block)
// step 2 is short; where it binds for most vectors the sequential walk dominates the stage.
#include <cooperative_groups.h>
#include <algorithm>
#include "common.cuh"
#include "feistel.cuh"
#include "tc05.cuh"

namespace cg = cooperative_groups;

namespace muse {

constexpr int kSkThreads = 512, kSkBatch = 64, kSkChunk = 64, kSkMaxCluster = 8;

template <int D> constexpr size_t stream_smem_bytes(int C) {
  return (size_t)(2 * kSkBatch * (D + 4) + 2 * C + kSkBatch * 32 + 2 * kSkMaxCluster * kSkBatch) * sizeof(float) +
         (size_t)(kSkBatch * 32 + 2 * kSkMaxCluster * kSkBatch + kSkBatch) * sizeof(int);
}

// One problem = one thread-block cluster of CS CTAs (CS = 1, 2, 4 or 8).  Every CTA holds the whole minibatch but
// only its own slice of the centroids: it computes the distances to that slice, the CTAs exchange their 64 best
// (distance, centroid) pairs through distributed shared memory, every CTA takes the overall arg-min, and each
// updates the centroids it owns.  A centroid row is only ever read and written by its owner, so the only traffic
// between the CTAs is the exchange, ordered by one hardware cluster barrier per minibatch.
template <class T, int D>
__global__ void __launch_bounds__(kSkThreads)
k_stream_kmeans(const T* __restrict__ X, int N, int C, uint64_t seed, int kind, float beta, int first_batch, int n_batches,
                float* __restrict__ totals, float* __restrict__ counts, float* __restrict__ centres,
                int32_t* __restrict__ assign_stream) {
  constexpr int LD = D + 4, EPL = D / 32, NW = kSkThreads / 32, PPW = kSkBatch / NW;
  constexpr int RV = D / 32;                   // 16-byte-of-fp32 groups of a row per loading thread (8 threads per row)
  cg::cluster_group cluster = cg::this_cluster();
  const int CS = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  extern __shared__ __align__(16) float sk_smem[];
  float* Xs = sk_smem;                         // [64][LD]  the minibatch
  float* Ct = Xs + kSkBatch * LD;              // [64][LD]  a chunk of centroids
  float* cn = Ct + kSkChunk * LD;              // [C] squared norms of the current centroids (own slice in use)
  float* cc = cn + C;                          // [C] counts c_j (own slice in use)
  float* bd = cc + C;                          // [64][32] per-thread best distances
  float* exd = bd + kSkBatch * 32;             // [2][CS max][64] exchanged best distances, double-buffered by step parity
  int* bi = reinterpret_cast<int*>(exd + 2 * kSkMaxCluster * kSkBatch);   // [64][32] centroids of bd
  int* exi = bi + kSkBatch * 32;               // [2][CS max][64] exchanged best centroids
  int* as = exi + 2 * kSkMaxCluster * kSkBatch;   // [64] the minibatch's assignments
  const int prob = blockIdx.x / CS, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const T* Xp = X + (size_t)prob * N * D;
  float* Tp = totals + (size_t)prob * C * D;
  float* Cp = centres + (size_t)prob * C * D;
  float* cntp = counts + (size_t)prob * C;
  const uint64_t strm = (uint64_t)prob * 2 + kind;
  const int per = ((C + CS - 1) / CS + 1) & ~1;                     // centroids per CTA (even: a thread takes two)
  const int j0 = min(C, rank * per), j1 = min(C, j0 + per);

  // state before the first minibatch of this call: the strided start (t = x, c = 1), or the caller's (t, c)
  for (int j = j0 + warp; j < j1; j += NW) {
    float t[EPL], c;
    if (first_batch == 0) {
      const int u = feistel_permute(j * (N / C), N, seed, strm);
      ldv<EPL>(Xp + (size_t)u * D + lane * EPL, t);
      c = 1.f;
      stv<EPL>(Tp + (size_t)j * D + lane * EPL, t);
    } else {
      ldv<EPL>(Tp + (size_t)j * D + lane * EPL, t);
      c = cntp[j];
    }
    float n2 = 0.f;
#pragma unroll
    for (int e = 0; e < EPL; ++e) { t[e] = t[e] / c; n2 = fmaf(t[e], t[e], n2); }
    stv<EPL>(Cp + (size_t)j * D + lane * EPL, t);
    n2 = warp_sum(n2);
    if (lane == 0) { cn[j] = n2; cc[j] = c; }
  }

  // rows of the next minibatch travel in registers while the current one is worked on: thread = (row, eighth of the row)
  const int lr = tid >> 3, lq = tid & 7;
  float4 xr[RV];
  auto fetch = [&](int s) {
    const int pos = s * kSkBatch + lr;
    const int u = pos < N ? feistel_permute(pos, N, seed, strm) : -1;
#pragma unroll
    for (int v = 0; v < RV; ++v)
      xr[v] = (u >= 0 && MUSE_IN_RANGE(u, N)) ? ld4(Xp + (size_t)u * D + (lq * RV + v) * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
  };
  if (n_batches > 0) fetch(first_batch);
  cluster.sync();                              // every CTA of the problem is running before any of them writes into another's shared memory

  // Thread tile: 4 vectors x 2 centroids of a 64 x 64 chunk.  A warp covers 8 vector rows x 4 centroid pairs at a
  // time, so that a shared-memory load of the warp touches 8 (vectors) or 4 (centroids) distinct rows: one wavefront each.
  const int pi = (warp & 1) * 32 + (lane & 7), ci = (warp >> 1) * 4 + (lane >> 3);   // vectors pi + 8 i; centroids 2 ci, 2 ci + 1
  for (int s = first_batch; s < first_batch + n_batches; ++s) {
    const int nb = min(kSkBatch, N - s * kSkBatch), par = s & 1;
#pragma unroll
    for (int v = 0; v < RV; ++v) *reinterpret_cast<float4*>(Xs + lr * LD + (lq * RV + v) * 4) = xr[v];
    if (s + 1 < first_batch + n_batches) fetch(s + 1);
    float best[4];
    int bidx[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) { best[i] = INFINITY; bidx[i] = 0x7fffffff; }
    for (int c0 = j0; c0 < j1; c0 += kSkChunk) {
      __syncthreads();                         // the minibatch is in place / the previous chunk has been used
      for (int e = tid; e < kSkChunk * (D / 4); e += kSkThreads) {
        const int r = e / (D / 4), q = e % (D / 4);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (c0 + r < j1) v = *reinterpret_cast<const float4*>(Cp + (size_t)(c0 + r) * D + q * 4);
        *reinterpret_cast<float4*>(Ct + r * LD + q * 4) = v;
      }
      __syncthreads();
      float acc[4][2];
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[i][0] = acc[i][1] = 0.f;
#pragma unroll 4
      for (int d4 = 0; d4 < D; d4 += 4) {
        const float4 a0 = *reinterpret_cast<const float4*>(Ct + (2 * ci) * LD + d4);
        const float4 a1 = *reinterpret_cast<const float4*>(Ct + (2 * ci + 1) * LD + d4);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 x = *reinterpret_cast<const float4*>(Xs + (pi + 8 * i) * LD + d4);
          acc[i][0] = fmaf(x.x, a0.x, fmaf(x.y, a0.y, fmaf(x.z, a0.z, fmaf(x.w, a0.w, acc[i][0]))));
          acc[i][1] = fmaf(x.x, a1.x, fmaf(x.y, a1.y, fmaf(x.z, a1.z, fmaf(x.w, a1.w, acc[i][1]))));
        }
      }
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int j = c0 + 2 * ci + k;
        if (j < j1) {
          const float n2 = cn[j];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float dist = fmaf(-2.f, acc[i][k], n2);           // |c|^2 - 2 x.c: |x|^2 is the same for every centroid
            if (dist < best[i]) { best[i] = dist; bidx[i] = j; }    // (ascending j: ties stay with the lower index)
          }
        }
      }
    }
    if (j0 >= j1) __syncthreads();             // (a CTA without centroids still has to have the minibatch in place)
#pragma unroll
    for (int i = 0; i < 4; ++i) { bd[(pi + 8 * i) * 32 + ci] = best[i]; bi[(pi + 8 * i) * 32 + ci] = bidx[i]; }
    __syncthreads();
    for (int k = 0; k < PPW; ++k) {            // a warp reduces four vectors' 32 candidates and posts the result to every CTA
      const int p = warp * PPW + k;
      float dv = bd[p * 32 + lane];
      int iv = bi[p * 32 + lane];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float od = __shfl_xor_sync(0xffffffffu, dv, o);
        const int oi = __shfl_xor_sync(0xffffffffu, iv, o);
        if (od < dv || (od == dv && oi < iv)) { dv = od; iv = oi; }
      }
      if (lane < CS) {
        *cluster.map_shared_rank(exd + (par * kSkMaxCluster + rank) * kSkBatch + p, lane) = dv;
        *cluster.map_shared_rank(exi + (par * kSkMaxCluster + rank) * kSkBatch + p, lane) = iv;
      }
    }
    cluster.sync();                            // every CTA's candidates have arrived (and the previous step's have been read)
    if (tid < kSkBatch) {
      float dv = exd[(par * kSkMaxCluster) * kSkBatch + tid];
      int iv = exi[(par * kSkMaxCluster) * kSkBatch + tid];
      for (int r = 1; r < CS; ++r) {
        const float od = exd[(par * kSkMaxCluster + r) * kSkBatch + tid];
        const int oi = exi[(par * kSkMaxCluster + r) * kSkBatch + tid];
        if (od < dv || (od == dv && oi < iv)) { dv = od; iv = oi; }
      }
      as[tid] = (tid < nb && (unsigned)iv < (unsigned)C) ? iv : (tid < nb ? 0 : -1);   // (a NaN row goes to centroid 0)
    }
    __syncthreads();
    // update: the first vector of the minibatch on a centroid ("leader") replays all of that centroid's vectors in order
    const int a_lo = as[lane], a_hi = as[lane + 32];                // the minibatch's assignments, two per lane
    for (int k = 0; k < PPW; ++k) {
      const int p = warp + NW * k;
      const int j = as[p];
      if (j < j0 || j >= j1) continue;                              // (warp-uniform: shared-memory values) not this CTA's centroid
      // the vectors of the minibatch on centroid j, as a 64-bit mask in stream order
      const unsigned long long mem = (unsigned long long)__ballot_sync(0xffffffffu, a_lo == j) |
                                     ((unsigned long long)__ballot_sync(0xffffffffu, a_hi == j) << 32);
      if (__ffsll((long long)mem) - 1 != p) continue;               // not the centroid's first vector
      float t[EPL], c = cc[j];
      ldv<EPL>(Tp + (size_t)j * D + lane * EPL, t);
      for (unsigned long long rest = mem; rest != 0ull; rest &= rest - 1ull) {
        const int q = __ffsll((long long)rest) - 1;
#pragma unroll
        for (int e = 0; e < EPL; ++e) t[e] = fmaf(beta, t[e], Xs[q * LD + lane * EPL + e]);
        c = fmaf(beta, c, 1.f);
      }
      stv<EPL>(Tp + (size_t)j * D + lane * EPL, t);
      float n2 = 0.f;
#pragma unroll
      for (int e = 0; e < EPL; ++e) { t[e] = t[e] / c; n2 = fmaf(t[e], t[e], n2); }
      stv<EPL>(Cp + (size_t)j * D + lane * EPL, t);
      n2 = warp_sum(n2);
      if (lane == 0) { cn[j] = n2; cc[j] = c; }
    }
    if (rank == 0 && assign_stream != nullptr && tid < nb) assign_stream[(size_t)prob * N + (size_t)s * kSkBatch + tid] = as[tid];
    __syncthreads();                           // the centroid rows written above are read by every thread in the next step
  }
  for (int j = j0 + tid; j < j1; j += kSkThreads) cntp[j] = cc[j];
  cluster.sync();                              // no CTA leaves while another may still write into its shared memory
}

// ---------------------------------------------------------------------------------------------
// The same pass with the distance product on the tensor cores (bf16 inputs, C <= 256 centroids per CTA), both sides of
// a clustering in one launch.  A CTA keeps ITS centroids resident in shared memory as bf16 hi + lo tiles
// ([128 centroids][D], 128-byte swizzle, K-major) and rewrites the rows it updates in place; their fp32 totals and counts
// stay in shared memory too where they fit.  The A operand is one [128][D] tile whose halves hold the current and the
// next minibatch: the product x.c of all 128 rows lands in tensor memory (tcgen05.mma, M = 128, N = 128, hi then lo
// accumulated) and only the current half's lanes are read.
//
// Bound by the latency of one step, N / 64 of them in a chain, so everything that a step does not need from the one
// before it is done elsewhere: four gather warps compute the shuffled positions and bring in the next minibatch by
// asynchronous copies; sixteen compute warps read the distances (every second pair of warps a half's 64 rows, a quarter
// of a tile's columns each) and post one candidate per quarter; two of them take the best of a vector's candidates, and all update the
// centroids whose first vector falls to them (a group of D / 8 lanes per vector).  Three barriers per step, the second a cluster
// barrier when a problem's centroids are spread over several CTAs.  Totals stay in shared memory and centre rows leave for global
// memory once, at the end.  Measured at 32 + 32 problems of 65536 vectors, D = 64, 128 centroids: 5.4 us per step and one side
// after the other (11.15 ms) at first, 3.6 us per step for both with two CTAs a problem and every warp taking the best candidates of all
// 64 vectors (16 warps of 130 instructions, on the step's path), 3.1 us now.  A step: products 1100 cycles, arg-min 1300, barriers
// 500, candidates 400, update 2500 (four groups' ballots, members in order, eight divisions, |c|^2 by shuffles).  Slower: divisions by a
// reciprocal and two corrections (3.4 us), columns as immediates in the arg-min with all norms loaded first (3.3 us).
// ---------------------------------------------------------------------------------------------
constexpr int kStCompute = 512, kStGather = 128, kStThreads = kStCompute + kStGather;

struct StSide {
  const __nv_bfloat16* X;
  float *totals, *counts, *centres;
  int32_t* assign_stream;
  int problems, C, kind, NT, tot_shared;     // NT: tiles of 128 centroids per CTA; tot_shared: totals resident in shared memory
};
struct StArgs { StSide s[2]; int N, first_batch, n_batches; float beta; uint64_t seed; };

template <int D> size_t stream_tc_smem_bytes(int NT, int tot_shared) {
  return 1024 + (size_t)(1 + 2 * NT) * 128 * D * 2 + (size_t)2 * NT * 128 * sizeof(float) + (tot_shared ? (size_t)NT * 128 * D * sizeof(float) : 0);
}

// running arg-min over W consecutive columns of tensor memory, four chains (columns mod 4)
template <int W>
__device__ __forceinline__ void st_argmin(uint32_t taddr, const float* cn, int j, float (&best)[4], int (&bidx)[4]) {
  float v[W];
  if constexpr (W == 32) tc::tmem_ld32(taddr, v);
  else if constexpr (W == 16) tc::tmem_ld16(taddr, v);
  else tc::tmem_ld8(taddr, v);
#pragma unroll
  for (int k = 0; k < W; k += 4) {
    const float4 n4 = *reinterpret_cast<const float4*>(cn + k);
    argmin_step(fmaf(-2.f, v[k], n4.x), j + k, best[0], bidx[0]);
    argmin_step(fmaf(-2.f, v[k + 1], n4.y), j + k + 1, best[1], bidx[1]);
    argmin_step(fmaf(-2.f, v[k + 2], n4.z), j + k + 2, best[2], bidx[2]);
    argmin_step(fmaf(-2.f, v[k + 3], n4.w), j + k + 3, best[3], bidx[3]);
  }
}

template <int D>
__global__ void __launch_bounds__(kStThreads, 1)
k_stream_kmeans_tc(const __grid_constant__ StArgs g, int* __restrict__ status) {
  typedef __nv_bfloat16 bf16;
  constexpr int EPL = D / 32, NW = kStCompute / 32, PPW = kSkBatch / NW, CPR = D / 8, kTile = 128 * D * 2;
  constexpr int LPG = D / 8, GPW = 32 / LPG;                 // update: lanes per centroid, centroids per warp at a time
  cg::cluster_group cluster = cg::this_cluster();
  const int CS = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  extern __shared__ __align__(1024) unsigned char st_raw[];
  __shared__ uint64_t sdone;
  __shared__ uint32_t tbase_s;
  __shared__ int2 cand[2][4 * kSkMaxCluster][kSkBatch];      // (distance bits, centroid) by step parity, CTA and column quarter
  __shared__ int pos_s[kSkBatch], as_s[kSkBatch];            // positions of the next minibatch, assignments of this one
  unsigned char* sm = st_raw + ((1024u - (tc::smem_u32(st_raw) & 1023u)) & 1023u);
  int prob = blockIdx.x / CS;
  const bool second = prob >= g.s[0].problems;
  const StSide& sd = g.s[second ? 1 : 0];
  if (second) prob -= g.s[0].problems;
  const int N = g.N, C = sd.C, NT = sd.NT, first_batch = g.first_batch, end_batch = g.first_batch + g.n_batches;
  const float beta = g.beta;
  unsigned char* Xs = sm;                                    // [128][D] bf16: two minibatches of 64 rows
  unsigned char* Chi = Xs + kTile;                           // NT tiles [128][D] bf16: high parts of this CTA's centroids
  unsigned char* Clo = Chi + (size_t)NT * kTile;             // ... and low parts
  float* cn = reinterpret_cast<float*>(Clo + (size_t)NT * kTile);   // [NT * 128] |c|^2 (infinity past the slice)
  float* cc = cn + NT * 128;                                 // [NT * 128] counts
  float* ts = cc + NT * 128;                                 // [NT * 128][D] totals (tot_shared)
  const int tid = threadIdx.x, warp = tc::warp_index(), lane = tid & 31;
  const bf16* Xp = sd.X + (size_t)prob * N * D;
  float* Tp = sd.totals + (size_t)prob * C * D;
  float* Cp = sd.centres + (size_t)prob * C * D;
  float* cntp = sd.counts + (size_t)prob * C;
  const uint64_t strm = (uint64_t)prob * 2 + sd.kind;
  const int per = ((C + CS - 1) / CS + 1) & ~1;
  const int j0 = min(C, rank * per), j1 = min(C, j0 + per);
  const int TN = per <= 32 ? 32 : per <= 64 ? 64 : 128;      // centroids of a tile that take part in the products
  // byte offset of elements [lane * EPL, lane * EPL + EPL) of row r inside a swizzled [128][D] tile
  const int e0 = lane * EPL, e8 = (lane % LPG) * 8;
  auto row_off = [&](int r) { return (uint32_t)((e0 >> 6) * 128 * 128) + tc::sw128_off(r, (e0 >> 3) & 7) + (uint32_t)((e0 & 7) * 2); };
  float* tot = sd.tot_shared ? ts : Tp + (size_t)j0 * D;     // row jl of this CTA's slice

  int tcols = 128;
  while (tcols < NT * 128) tcols *= 2;
  if (warp == 0) tc::tmem_alloc(&tbase_s, tcols);
  if (tid == 0) { tc::mbar_init(&sdone, 1); tc::mbar_init_fence(); }
  for (int e = tid; e < (1 + 2 * NT) * kTile / 16; e += kStThreads) reinterpret_cast<uint4*>(sm)[e] = make_uint4(0u, 0u, 0u, 0u);
  for (int e = tid; e < NT * 128; e += kStThreads) { cn[e] = INFINITY; cc[e] = 0.f; }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tbase = tbase_s;
  pdl_wait();
  pdl_trigger();

  // a centroid row from its totals: bf16 hi / lo into the resident tiles, |c|^2 and count
  auto put_centroid = [&](int jl, float (&t)[EPL], float c) {
    float n2 = 0.f;
    uint32_t hw[EPL / 2], lw[EPL / 2];
#pragma unroll
    for (int e = 0; e < EPL; ++e) { t[e] = t[e] / c; n2 = fmaf(t[e], t[e], n2); }
#pragma unroll
    for (int e = 0; e < EPL; e += 2) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(t[e], t[e + 1]);
      const __nv_bfloat162 l = __floats2bfloat162_rn(t[e] - __low2float(h), t[e + 1] - __high2float(h));
      hw[e / 2] = *reinterpret_cast<const uint32_t*>(&h);
      lw[e / 2] = *reinterpret_cast<const uint32_t*>(&l);
    }
    const uint32_t off = (uint32_t)(jl >> 7) * kTile + row_off(jl & 127);
    if (EPL == 4) {
      *reinterpret_cast<uint2*>(Chi + off) = make_uint2(hw[0], hw[EPL / 2 - 1]);
      *reinterpret_cast<uint2*>(Clo + off) = make_uint2(lw[0], lw[EPL / 2 - 1]);
    } else {
      *reinterpret_cast<uint32_t*>(Chi + off) = hw[0];
      *reinterpret_cast<uint32_t*>(Clo + off) = lw[0];
    }
    n2 = warp_sum(n2);
    if (lane == 0) { cn[jl] = n2; cc[jl] = c; }
  };

  for (int j = j0 + warp; j < j1; j += kStThreads / 32) {
    float t[EPL], c;
    if (first_batch == 0) {
      const int u = feistel_permute(j * (N / C), N, g.seed, strm);
      ldv<EPL>(Xp + (size_t)u * D + e0, t);
      c = 1.f;
    } else {
      ldv<EPL>(Tp + (size_t)j * D + e0, t);
      c = cntp[j];
    }
    stv<EPL>(tot + (size_t)(j - j0) * D + e0, t);
    put_centroid(j - j0, t, c);
  }

  // gather warps: the rows of minibatch s into half s & 1 of the X tile; positions one minibatch ahead
  const int gt = tid - kStCompute;
  int pos_n = -1;
  auto position = [&](int s) {
    const int pos = s * kSkBatch + gt;
    return gt >= 0 && gt < kSkBatch && s < end_batch && pos < N ? feistel_permute(pos, N, g.seed, strm) : -1;
  };
  auto gather = [&](int s) {
    if (gt < kSkBatch) pos_s[gt] = pos_n;
    tc::named_bar_sync(2, kStGather);
    for (int e = gt; e < kSkBatch * CPR; e += kStGather) {
      const int r = e / CPR, c = e % CPR, u = pos_s[r];
      const bool in = u >= 0 && MUSE_IN_RANGE(u, N);
      const int n = in ? 16 : 0;                             // 0 source bytes: the 16 bytes are zero-filled
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                   ::"r"(tc::smem_u32(Xs + (c >> 3) * 128 * 128 + tc::sw128_off((s & 1) * 64 + r, c & 7))),
                     "l"(Xp + (size_t)(in ? u : 0) * D + c * 8), "r"(n) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    pos_n = position(s + 1);
    if (pos_n >= 0)                                          // have the rows of the minibatch after this one on their way
#pragma unroll
      for (int o = 0; o < D * 2; o += 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char*>(Xp + (size_t)pos_n * D) + o));
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    tc::named_bar_sync(2, kStGather);                        // pos_s may be rewritten
  };
  if (gt >= 0) { pos_n = position(first_batch); if (g.n_batches > 0) gather(first_batch); }
  tc::fence_async_smem();
  cluster.sync();                                            // every CTA of the problem is running before any of them writes into another's shared memory
  bool ok = true;
  const uint32_t idesc = tc::idesc_bf16(128, TN, 0, 0);
  const uint64_t dx0 = tc::smem_desc_sw128(tc::smem_u32(Xs), 16, 1024), dh0 = tc::smem_desc_sw128(tc::smem_u32(Chi), 16, 1024),
                 dl0 = tc::smem_desc_sw128(tc::smem_u32(Clo), 16, 1024);

  for (int s = first_batch, it = 0; s < end_batch; ++s, ++it) {
    const int nb = min(kSkBatch, N - s * kSkBatch), par = s & 1;
    tc::fence_before_sync();
    __syncthreads();                                         // A: the minibatch and the rewritten centroid rows are in place
    if (gt >= 0) {
      if (s + 1 < end_batch) { gather(s + 1); tc::fence_async_smem(); }
      if (CS > 1) cluster.sync();
      continue;
    }
    if (warp == 0) {                                         // ---- products
      tc::fence_after_sync();
      for (int t = 0; t < NT; ++t) {
        const uint64_t dh = tc::desc_step(dh0, (uint32_t)t * kTile), dl = tc::desc_step(dl0, (uint32_t)t * kTile);
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks)
          tc::mma_bf16_ss_warp(tbase + t * 128, tc::desc_step(dx0, (ks / 4) * 128 * 128 + (ks % 4) * 32),
                               tc::desc_step(dh, (ks / 4) * 128 * 128 + (ks % 4) * 32), idesc, ks > 0);
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks)
          tc::mma_bf16_ss_warp(tbase + t * 128, tc::desc_step(dx0, (ks / 4) * 128 * 128 + (ks % 4) * 32),
                               tc::desc_step(dl, (ks / 4) * 128 * 128 + (ks % 4) * 32), idesc, 1);
      }
      tc::mma_commit_warp(&sdone);
    }
    if (((warp & 3) >> 1) == par) {                          // ---- arg-min: thread = (vector, 32 columns of every tile)
      if (ok && !tc::mbar_wait(&sdone, it & 1)) ok = false;
      tc::fence_after_sync();
      const uint32_t tl = tbase + ((uint32_t)((warp & 3) * 32) << 16);
      const int quarter = warp >> 2;
      float best[4];
      int bidx[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) { best[e] = INFINITY; bidx[e] = 0x7fffffff; }
      for (int t = 0; t < NT; ++t) {
        const int c0 = t * 128 + quarter * (TN / 4);
        if (TN == 128) st_argmin<32>(tl + c0, cn + c0, j0 + c0, best, bidx);
        else if (TN == 64) st_argmin<16>(tl + c0, cn + c0, j0 + c0, best, bidx);
        else st_argmin<8>(tl + c0, cn + c0, j0 + c0, best, bidx);
      }
      tc::fence_before_sync();
#pragma unroll
      for (int e = 1; e < 4; ++e) argmin_tie_step(best[e], bidx[e], best[0], bidx[0]);
      const int p = (warp & 1) * 32 + lane;
      const int2 mine = make_int2(__float_as_int(best[0]), bidx[0]);
      if (CS == 1) cand[par][quarter][p] = mine;
      else
        for (int r = 0; r < CS; ++r) *cluster.map_shared_rank(&cand[par][rank * 4 + quarter][p], r) = mine;
    }
    if (CS == 1) tc::named_bar_sync(1, kStCompute); else cluster.sync();     // B: every candidate has arrived
    // two warps: the minibatch's assignments (lower distance wins, the lower centroid on a tie); every warp then holds all, two per lane
    if (tid < kSkBatch) {
      float dv = INFINITY;
      int iv = 0x7fffffff;
#pragma unroll 4
      for (int r = 0; r < 4 * CS; ++r) argmin_tie_step(__int_as_float(cand[par][r][tid].x), cand[par][r][tid].y, dv, iv);
      as_s[tid] = tid < nb ? ((unsigned)iv < (unsigned)C ? iv : 0) : -1;     // (a NaN row goes to centroid 0)
    }
    tc::named_bar_sync(1, kStCompute);
    const int a_lo = as_s[lane], a_hi = as_s[lane + 32];
    // update: the first vector of the minibatch on a centroid replays all of that centroid's vectors in stream order.
    // A group of D / 8 lanes takes a vector (8 dims per lane), so a warp works on several centroids at once.
#pragma unroll
    for (int k0 = 0; k0 < PPW; k0 += GPW) {
      int j = -1, mlo = 0, mhi = 0;
#pragma unroll
      for (int k = 0; k < GPW; ++k) {
        const int p = warp * PPW + k0 + k;
        const int jk = __shfl_sync(0xffffffffu, p < 32 ? a_lo : a_hi, p & 31);
        const unsigned lo = __ballot_sync(0xffffffffu, a_lo == jk), hi = __ballot_sync(0xffffffffu, a_hi == jk);
        const bool first = p < 32 ? (lo & ((1u << p) - 1u)) == 0u : lo == 0u && (hi & ((1u << (p - 32)) - 1u)) == 0u;
        if (lane / LPG == k && first && jk >= j0 && jk < j1) { j = jk; mlo = (int)lo; mhi = (int)hi; }
      }
      if (!__any_sync(0xffffffffu, j >= 0)) continue;
      const bool mine = j >= 0;                              // else not this CTA's centroid, or not its first vector
      const int jl = mine ? j - j0 : 0;
      float* tr = tot + (size_t)jl * D + e8;
      float t[8], c = cc[jl];
      {
        const float4 x = *reinterpret_cast<const float4*>(tr), y = *reinterpret_cast<const float4*>(tr + 4);
        t[0] = x.x; t[1] = x.y; t[2] = x.z; t[3] = x.w; t[4] = y.x; t[5] = y.y; t[6] = y.z; t[7] = y.w;
      }
      for (unsigned long long rest = ((unsigned long long)(unsigned)mhi << 32) | (unsigned)mlo; rest != 0ull; rest &= rest - 1ull) {
        const int q = par * 64 + __ffsll((long long)rest) - 1;
        const uint4 u = *reinterpret_cast<const uint4*>(Xs + (e8 >> 6) * 128 * 128 + tc::sw128_off(q, (e8 >> 3) & 7));
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          t[2 * e] = fmaf(beta, t[2 * e], __uint_as_float(w[e] << 16));
          t[2 * e + 1] = fmaf(beta, t[2 * e + 1], __uint_as_float(w[e] & 0xffff0000u));
        }
        c = fmaf(beta, c, 1.f);
      }
      __syncwarp();
      if (mine) {
        *reinterpret_cast<float4*>(tr) = make_float4(t[0], t[1], t[2], t[3]);
        *reinterpret_cast<float4*>(tr + 4) = make_float4(t[4], t[5], t[6], t[7]);
      }
      uint32_t hw[4], lw[4];
      float n2[8 / EPL];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        t[e] = t[e] / c;
        n2[e / EPL] = e % EPL == 0 ? t[e] * t[e] : fmaf(t[e], t[e], n2[e / EPL]);
      }
#pragma unroll
      for (int e = 0; e < 8; e += 2) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(t[e], t[e + 1]);
        const __nv_bfloat162 l = __floats2bfloat162_rn(t[e] - __low2float(h), t[e + 1] - __high2float(h));
        hw[e / 2] = *reinterpret_cast<const uint32_t*>(&h);
        lw[e / 2] = *reinterpret_cast<const uint32_t*>(&l);
      }
      // |c|^2 in the order of put_centroid's reduction (EPL dims per lane of a whole warp, butterfly from 16 down)
#pragma unroll
      for (int o = LPG / 2; o > 0; o >>= 1)
#pragma unroll
        for (int e = 0; e < 8 / EPL; ++e) n2[e] += __shfl_xor_sync(0xffffffffu, n2[e], o);
      if (8 / EPL == 4) { n2[0] += n2[8 / EPL - 2]; n2[1] += n2[8 / EPL - 1]; }
      n2[0] += n2[1];
      if (mine) {
        const uint32_t off = (uint32_t)(jl >> 7) * kTile + (uint32_t)((e8 >> 6) * 128 * 128) + tc::sw128_off(jl & 127, (e8 >> 3) & 7);
        *reinterpret_cast<uint4*>(Chi + off) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
        *reinterpret_cast<uint4*>(Clo + off) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
        if (lane % LPG == 0) { cn[jl] = n2[0]; cc[jl] = c; }
      }
      __syncwarp();
    }
    if (rank == 0 && sd.assign_stream != nullptr && warp == NW - 1) {
      int32_t* as = sd.assign_stream + (size_t)prob * N + (size_t)s * kSkBatch;
      if (lane < nb) as[lane] = a_lo;
      if (lane + 32 < nb) as[lane + 32] = a_hi;
    }
    tc::fence_async_smem();                                  // the rewritten centroid rows are read by the tensor cores
  }
  __syncthreads();
  for (int j = j0 + warp; j < j1; j += kStThreads / 32) {     // totals, counts and centres leave once
    float t[EPL];
    const float c = cc[j - j0];
    ldv<EPL>(tot + (size_t)(j - j0) * D + e0, t);
    if (sd.tot_shared) stv<EPL>(Tp + (size_t)j * D + e0, t);
#pragma unroll
    for (int e = 0; e < EPL; ++e) t[e] = t[e] / c;
    stv<EPL>(Cp + (size_t)j * D + e0, t);
    if (lane == 0) cntp[j] = c;
  }
  if (!ok && lane == 0) report_status(status, MUSE_STATUS_ASSIGN_TIMEOUT);
  tc::fence_before_sync();
  cluster.sync();                                            // no CTA leaves while another may still write into its shared memory
  if (warp == 0) tc::tmem_dealloc(tbase, tcols);
}

// bf16 sides with at most 256 * 8 centroids: one launch of k_stream_kmeans_tc over all of their problems.
template <int D>
static int stream_kmeans_tc(const Dims& d, const StreamSide* sides, int n, uint64_t seed, float beta, int first_batch, int n_batches,
                            int* status, cudaStream_t st) {
  StArgs g = {};
  g.N = d.N; g.first_batch = first_batch; g.n_batches = n_batches; g.beta = beta; g.seed = seed;
  int problems = 0, C = 0;
  for (int k = 0; k < n; ++k) { problems += sides[k].problems; C = sides[k].C > C ? sides[k].C : C; }
  // CTAs per problem: at most 256 centroids (two tiles) per CTA; from 256 per CTA on twice the CTAs, as long as every CTA still has an SM
  // of its own.  (A cluster barrier and the exchange of candidates cost more than half as many columns of an arg-min: us a step, lines at
  // 64 | 128 | 256 | 512 centroids: 64 problems of 128 centroids, D = 64 3.70 | 3.69 | 3.31 | 3.32, D = 128 6.53 | 6.53 | 5.46 | 5.46; 2 of 64
  // and 128 5.28 | 5.00 | 3.65 | 3.65; 20 of 152 and 256 3.96 | 3.96 | 3.79 | 3.90; 8 of 64 and 256, D = 128 6.14 | 5.35 | 5.24 | 5.47.)
  int cs = 1;
  while (cs < kSkMaxCluster && (C > 256 * cs || (C >= 256 * cs && (long long)problems * cs * 2 <= sm_count()))) cs *= 2;
  size_t smem = 0;
  for (int k = 0; k < n; ++k) {
    const StreamSide& s = sides[k];
    const int per = ((s.C + cs - 1) / cs + 1) & ~1, NT = (per + 127) / 128;
    const int shared = stream_tc_smem_bytes<D>(NT, 1) <= 200 * 1024;
    g.s[k] = StSide{(const __nv_bfloat16*)s.X, s.totals, s.counts, s.centres, s.assign_stream, s.problems, s.C, s.kind, NT, shared};
    const size_t b = stream_tc_smem_bytes<D>(NT, shared);
    smem = b > smem ? b : smem;
  }
  prof_mark("k_stream_kmeans_tc", st);
  return launch_pdl_cluster(k_stream_kmeans_tc<D>, dim3(problems * cs), kStThreads, smem, cs, st, g, status);
}

template <class T, int D>
static int stream_kmeans_ffma(const Dims& d, const StreamSide& s, uint64_t seed, float beta, int first_batch, int n_batches, cudaStream_t st) {
  const size_t smem = stream_smem_bytes<D>(s.C);
  // CTAs per problem: enough that a CTA owns at most two chunks of 64 centroids, as long as the GPU has room for them
  int cs = 1;
  while (cs < kSkMaxCluster && s.C > 2 * kSkChunk * cs && (long long)s.problems * cs * 2 <= 2 * sm_count()) cs *= 2;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cs; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.stream = st;
  cfg.gridDim = dim3(s.problems * cs);
  cfg.blockDim = dim3(kSkThreads);
  cfg.dynamicSmemBytes = smem;
  MUSE_CUDA_OK(cudaFuncSetAttribute(k_stream_kmeans<T, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  prof_mark("k_stream_kmeans", st);
  MUSE_CUDA_OK(cudaLaunchKernelEx(&cfg, k_stream_kmeans<T, D>, (const T*)s.X, d.N, s.C, seed, s.kind, beta, first_batch, n_batches, s.totals, s.counts,
                                  s.centres, s.assign_stream));
  return MUSE_OK;
}

int stream_kmeans(const Dims& d, int dtype, const StreamSide* sides, int n, uint64_t seed, float beta, int first_batch, int n_batches,
                  int32_t* status, cudaStream_t st) {
  const int all = cdiv(d.N, kSkBatch);
  if (first_batch < 0 || first_batch > all) return MUSE_ERR_INVALID_ARG;
  if (n_batches < 0) n_batches = all - first_batch;
  if (first_batch + n_batches > all) return MUSE_ERR_INVALID_ARG;
  StreamSide tc_sides[2];
  int ntc = 0;
  for (int k = 0; k < n; ++k) {
    const StreamSide& s = sides[k];
    if (dtype == MUSE_BF16 && s.C <= 256 * kSkMaxCluster) { tc_sides[ntc++] = s; continue; }
    if (dtype == MUSE_F32) MUSE_RC((d.D == 64 ? stream_kmeans_ffma<float, 64> : stream_kmeans_ffma<float, 128>)(d, s, seed, beta, first_batch, n_batches, st));
    else MUSE_RC((d.D == 64 ? stream_kmeans_ffma<__nv_bfloat16, 64> : stream_kmeans_ffma<__nv_bfloat16, 128>)(d, s, seed, beta, first_batch, n_batches, st));
  }
  if (ntc == 0) return MUSE_OK;
  return (d.D == 64 ? stream_kmeans_tc<64> : stream_kmeans_tc<128>)(d, tc_sides, ntc, seed, beta, first_batch, n_batches, status, st);
}

// ---------------------------------------------------------------------------------------------
// Balanced assignment
// ---------------------------------------------------------------------------------------------

struct RankSide { const int32_t *assign, *off, *perm; int32_t *rank, *flags; int problems, C, cap; };
struct RankArgs { RankSide s[2]; int N, S, Bs; };

// rank of every vector inside its (block, cluster) bucket in position order (the sort is stable); flags names the
// 128-vector tiles that hold a displaced one
__global__ void __launch_bounds__(256)
k_bucket_rank(const __grid_constant__ RankArgs g) {
  const int N = g.N, pos = blockIdx.x * blockDim.x + threadIdx.x;
  int prob = blockIdx.y;
  const bool second = prob >= g.s[0].problems;
  const RankSide& sd = g.s[second ? 1 : 0];
  if (second) prob -= g.s[0].problems;
  pdl_wait();
  pdl_trigger();
  if (pos >= N) return;
  const int t = sd.perm[(size_t)prob * N + pos];
  if (!MUSE_IN_RANGE(t, N)) return;
  const int a = min(max(sd.assign[(size_t)prob * N + t], 0), sd.C - 1);
  const int key = (t / g.Bs) * sd.C + a;
  const int r = pos - sd.off[(size_t)prob * ((size_t)sd.C * g.S + 1) + key];
  sd.rank[(size_t)prob * N + t] = r;
  if (r >= sd.cap) sd.flags[(size_t)prob * cdiv(N, kAsgTile) + t / kAsgTile] = 1;
}

constexpr int kCapThreads = 512;

// Step 2: the displaced vectors of one (problem, block), in position order; each takes the nearest centroid whose bucket
// still has room.  The distances of every vector to every centroid were written by the step-1 assignment, so a placement is
// a masked arg-min over one row of that matrix (ties to the lower index).
__global__ void __launch_bounds__(kCapThreads)
k_cap_overflow(int N, int C, int S, int Bs, int cap, const float* dist, const int32_t* off, const int32_t* rank, int32_t* assign) {
  constexpr int NW = kCapThreads / 32;
  extern __shared__ int cap_smem[];
  int* size = cap_smem;                        // [C] bucket sizes of this block
  __shared__ int lst[kCapThreads], wcnt[NW], ri[NW];
  __shared__ float rd[NW];
  const int b = blockIdx.x, prob = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int32_t* o = off + (size_t)prob * (C * S + 1) + (size_t)b * C;
  const int32_t* rk = rank + (size_t)prob * N;
  int32_t* as = assign + (size_t)prob * N;
  pdl_wait();
  pdl_trigger();
  for (int j = tid; j < C; j += kCapThreads) size[j] = min(o[j + 1] - o[j], cap);     // step 1: the first cap of a bucket keep it
  __syncthreads();
  for (int base = b * Bs; base < (b + 1) * Bs; base += kCapThreads) {
    // the displaced vectors of this stretch, in position order
    const int t = base + tid;
    const bool over = t < (b + 1) * Bs && rk[t] >= cap;
    const unsigned bal = __ballot_sync(0xffffffffu, over);
    if (lane == 0) wcnt[warp] = __popc(bal);
    __syncthreads();
    int before = 0, total = 0;
    for (int w = 0; w < NW; ++w) { if (w < warp) before += wcnt[w]; total += wcnt[w]; }
    if (over) lst[before + __popc(bal & ((1u << lane) - 1u))] = t;
    __syncthreads();
    for (int e = 0; e < total; ++e) {
      const int u = lst[e];
      const float* dr = dist + ((size_t)prob * N + u) * C;
      float best = INFINITY;
      int bj = 0x7fffffff;
      for (int j = tid; j < C; j += kCapThreads) {
        if (size[j] >= cap) continue;
        const float dv = dr[j];
        if (dv < best) { best = dv; bj = j; }                          // (ascending j per thread)
      }
#pragma unroll
      for (int o2 = 16; o2 > 0; o2 >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, best, o2);
        const int oj = __shfl_xor_sync(0xffffffffu, bj, o2);
        if (ob < best || (ob == best && oj < bj)) { best = ob; bj = oj; }
      }
      if (lane == 0) { rd[warp] = best; ri[warp] = bj; }
      __syncthreads();
      if (tid == 0) {
        float bd = rd[0];
        int bi = ri[0];
        for (int w = 1; w < NW; ++w)
          if (rd[w] < bd || (rd[w] == bd && ri[w] < bi)) { bd = rd[w]; bi = ri[w]; }
        if ((unsigned)bi >= (unsigned)C)                               // every distance was NaN: first centroid with room
          for (bi = 0; bi < C - 1 && size[bi] >= cap; ++bi) {}
        as[u] = bi;
        size[bi] += 1;
      }
      __syncthreads();
    }
  }
}

// Scratch: each side's arrays, then one distance matrix that the sides use in turn.
struct BalancedWs { int32_t *status, *rank[2], *flags[2]; float* dist; };

static BalancedWs balanced_ws(const Dims& d, Arena& ar, LloydSide* s, int n) {
  BalancedWs w = {};
  size_t dist = 0;
  w.status = ar.take<int32_t>(kStatusWords);
  for (int k = 0; k < n; ++k) {
    lloyd_side_ws(d, ar, s[k]);
    w.rank[k] = ar.take<int32_t>((size_t)s[k].problems * d.N);
    w.flags[k] = ar.take<int32_t>((size_t)s[k].problems * cdiv(d.N, kAsgTile));
    dist = std::max(dist, (size_t)s[k].problems * d.N * s[k].C);
  }
  w.dist = ar.take<float>(dist);               // |c|^2 - 2 x.c of the tiles that hold displaced vectors
  return w;
}

size_t balanced_ws_bytes(const Dims& d, const int* problems, const int* C, int n) {
  Arena ar(nullptr);
  LloydSide s[2] = {};
  for (int k = 0; k < n; ++k) { s[k].problems = problems[k]; s[k].C = C[k]; }
  balanced_ws(d, ar, s, n);
  return ar.used;
}

int balanced_assign(const Dims& d, int dtype, const BalancedSide* sides, int n, float factor, void* ws, cudaStream_t st) {
  Arena ar(ws);
  LloydSide s[2] = {};
  for (int k = 0; k < n; ++k) {
    s[k].X = sides[k].X; s[k].problems = sides[k].problems; s[k].C = sides[k].C; s[k].kind = sides[k].kind;
    s[k].assign = sides[k].assign; s[k].centres = const_cast<float*>(sides[k].centres);
  }
  const BalancedWs w = balanced_ws(d, ar, s, n);
  // step 1: nearest centroid of every vector (the Lloyd path's final assignment against given centres)
  // (the entry points have cleared the status words; what the streaming pass reported there stays)
  MUSE_RC(lloyd(d, dtype, s, n, MUSE_INIT_CENTRES, 0, 0, false, w.status, st));
  // the sides whose cap can bind; for the others the nearest centroid is the answer
  SortSide sort[2];
  RankArgs r = {};
  LloydSide b[2] = {};
  int nb = 0, problems = 0;
  for (int k = 0; k < n; ++k) {
    const int cap = factor > 0.f ? (int)ceil((double)factor * d.Bs / s[k].C) : d.Bs;
    if (cap >= d.Bs) continue;
    MUSE_CUDA_OK(cudaMemsetAsync(w.flags[k], 0, (size_t)s[k].problems * cdiv(d.N, kAsgTile) * sizeof(int32_t), st));
    sort[nb] = SortSide{s[k].assign, s[k].off, s[k].perm, s[k].problems, s[k].C, 0};      // segments (block, cluster)
    r.s[nb] = RankSide{s[k].assign, s[k].off, s[k].perm, w.rank[k], w.flags[k], s[k].problems, s[k].C, cap};
    b[nb] = s[k];
    b[nb].dist = w.dist; b[nb].flags = w.flags[k];
    problems += s[k].problems;
    ++nb;
  }
  if (nb == 0) return MUSE_OK;
  MUSE_RC(bucket_sort(sort, nb, d.N, d.S, d.Bs, st));
  r.N = d.N; r.S = d.S; r.Bs = d.Bs;
  prof_mark("k_bucket_rank", st);
  MUSE_RC(launch_pdl(k_bucket_rank, dim3(cdiv(d.N, 256), problems), 256, 0, st, r));
  // step 2, where a bucket overflows: the distances of the tiles that hold displaced vectors, and the placements
  for (int k = 0; k < nb; ++k) {
    MUSE_RC(assign_distances(d, dtype, b[k], w.status, st));
    prof_mark("k_cap_overflow", st);
    MUSE_RC(launch_pdl(k_cap_overflow, dim3(d.S, r.s[k].problems), kCapThreads, (size_t)r.s[k].C * sizeof(int), st, d.N, r.s[k].C, d.S, d.Bs,
                       r.s[k].cap, b[k].dist, r.s[k].off, r.s[k].rank, b[k].assign));
  }
  return MUSE_OK;
}

}  // namespace muse
