// Spatial block selection and near field of the two-level retrieval (Section "Two-Level Retrieval", second level;
// Section "Output merging", component 2), the kernel for bf16 mode with at most 8 earlier blocks (S <= 9); the
// definitions are those at the head of block_select.cu, which serves the other shapes.
//
// A CTA takes the queries of one cluster i over all blocks, up to 256 at a time (bf16 rows in shared memory), and lists
// their (query, slot) pairs by selected cluster j.
//   1. A warp takes a cluster j, keeps the rows of its earlier blocks in registers and walks the list 16 pairs at a time:
//      S^T = kappa q^T, kappa_hi on rows 0-7 of the product and kappa_lo on rows 8-15 (mma.sync: 8 blocks by 16 gathered
//      pairs is far below the 64 rows of the smallest tcgen05 product); the logits go to shared memory.
//   2. A thread per pair makes the top-k2 choice.
//   3. A warp per query: the softmax over its stand-in logits, and the weighted nu rows, lanes sharing D.
// A lane per query, as step 1 was before, has work in two or three lanes of a warp: 32 queries of one segment rarely agree
// on a cluster.
//
// Bound: L2 reads of step 3 (128 bytes per pair and block at D = 64).  8 heads of two sequences of 64k tokens, D = 64,
// 128 x 128 clusters, 8 slots, 8 blocks: 4.35 ms with a lane per query, 2.32 ms.
#include <algorithm>
#include "common.cuh"
#include "near.cuh"

namespace muse {

typedef __nv_bfloat16 bf16;

constexpr int kBqMaxSB = kNbGroup;

template <int D> struct BqLay {
  static constexpr int kThreads = D == 128 ? 256 : 512, kQ = D == 128 ? 128 : 256;       // queries of a chunk at most
  static constexpr int LD = D + 8;                          // bf16 per query row
  static constexpr int oQ = 0, oG = oQ + kQ * LD * 2, oRow = oG + kNbPairs * kNbGroup * 4, oNb = oRow + kQ * 4, oList = oNb + kQ * 4,
                       oSel = oList + kNbPairs * 4, oOff = oSel + kNbPairs * 2;          // then Ck ints
};

bool block_select_q_supported(const Dims& d, int dtype) { return dtype == MUSE_BF16 && d.causal && d.SB <= kBqMaxSB && d.k2 <= 8; }

template <int D>
__global__ void __launch_bounds__(BqLay<D>::kThreads, 2)
k_block_select_q(Dims dm, const bf16* __restrict__ Q, const int32_t* __restrict__ off_q, const int32_t* __restrict__ perm_q,
                 const int32_t* __restrict__ sel, SummPtrs sp, const int32_t* __restrict__ bsel_in, int32_t* __restrict__ bsel_out,
                 float* __restrict__ o_near, float* __restrict__ lse_near) {
  pdl_wait();
  pdl_trigger();
  typedef BqLay<D> L;
  constexpr int kThreads = L::kThreads, kWarps = kThreads / 32, LD = L::LD, EPL = D / 32, KS = D / 16, G = kNbGroup;
  extern __shared__ __align__(16) unsigned char bq_smem[];
  const int m = dm.m, k2 = dm.k2, SB = dm.SB, Ck = dm.Ck;
  bf16* q_s = (bf16*)(bq_smem + L::oQ);
  float* lg_s = (float*)(bq_smem + L::oG);                           // [pair][8] stand-in logits; later weights
  int *row_s = (int*)(bq_smem + L::oRow), *nb_s = (int*)(bq_smem + L::oNb), *off = (int*)(bq_smem + L::oOff);
  uint32_t* list = (uint32_t*)(bq_smem + L::oList);                  // query << 16 | pair
  uint16_t* sel_s = (uint16_t*)(bq_smem + L::oSel);
  __shared__ int pre_s[kBqMaxSB + 2], p0_s[kBqMaxSB + 2], next_s;    // queries of the cluster before block b; where block b's start
  const int i = blockIdx.x, pq = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, n = lane >> 2, c = lane & 3;
  const int32_t* pm = perm_q + (size_t)pq * dm.N;
  const size_t estep = (size_t)dm.Cq * Ck;
  const size_t ebase = ((size_t)pq * SB * dm.Cq + i) * Ck;
  if (tid == 0) {
    const int32_t* oq = off_q + (size_t)pq * (dm.S * dm.Cq + 1) + i;
    int at = 0;
    for (int b = 0; b < dm.S; ++b) {                                 // S <= 9
      p0_s[b] = oq[(size_t)b * dm.Cq];
      pre_s[b] = at;
      at += oq[(size_t)b * dm.Cq + 1] - p0_s[b];
    }
    pre_s[dm.S] = at;
  }
  __syncthreads();
  const int total = pre_s[dm.S], QC = min(L::kQ, kNbPairs / m);
  for (int c0 = blockIdx.z * QC; c0 < total; c0 += gridDim.z * QC) {
    const int nq = min(QC, total - c0);
    // ---- the chunk's queries, their pairs, the list of pairs by selected cluster
    for (int r = tid; r < nq; r += kThreads) {
      int b = 0;
      while (pre_s[b + 1] <= c0 + r) ++b;
      int t = pm[p0_s[b] + c0 + r - pre_s[b]];
      if (!MUSE_IN_RANGE(t, dm.N)) t = -1;
      row_s[r] = t;
      nb_s[r] = b;
    }
    for (int j = tid; j < Ck; j += kThreads) off[j] = 0;
    if (tid == 0) next_s = 0;
    __syncthreads();
    constexpr int kP = D / 8;                                        // 16-byte pieces of a row
    for (int e = tid; e < nq * kP; e += kThreads) {
      const int r = e / kP, p = e % kP;
      nb_cp_async16(q_s + r * LD + p * 8, Q + ((size_t)pq * dm.N + max(row_s[r], 0)) * D + p * 8);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    for (int e = tid; e < nq * m; e += kThreads) {
      const int r = e / m, t = row_s[r];
      int j = -1;
      if (t >= 0 && nb_s[r] > 0) {
        j = sel[((size_t)pq * dm.N + t) * m + (e - r * m)];
        if (j < 0 || j >= Ck) j = -1;
      }
      sel_s[e] = (uint16_t)(j < 0 ? 0xffff : j);
      if (j >= 0) atomicAdd(&off[j], 1);
      float4* lg = reinterpret_cast<float4*>(lg_s + e * G);
      lg[0] = lg[1] = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    }
    __syncthreads();
    if (warp == 0) nb_scan(off, Ck, lane);
    __syncthreads();
    for (int e = tid; e < nq * m; e += kThreads) {
      const int j = sel_s[e];
      if (j != 0xffff) list[atomicAdd(&off[j], 1)] = (uint32_t)(e / m) << 16 | (uint32_t)e;   // off[j]: then the end of j's pairs
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    const int nbmax = nb_s[nq - 1];                                  // queries go by block
    __syncthreads();

    // ---- step 1.  Lane (n, c) holds block n's dims c D/4 .. of kappa: the k index of a product is a permutation of D, the
    // same for both operands, so that a lane's operands are 16-byte loads.
    for (;;) {
      int j = 0;
      if (lane == 0) j = atomicAdd(&next_s, 1);
      j = __shfl_sync(0xffffffffu, j, 0);
      if (j >= Ck) break;
      const int o0 = j > 0 ? off[j - 1] : 0, o1 = off[j];
      if (o0 == o1) continue;
      const size_t ent = ebase + (size_t)n * estep + j;
      const bool here = n < nbmax;
      uint4 kh[KS / 2], kl[KS / 2];
#pragma unroll
      for (int t = 0; t < KS / 2; ++t) {
        const size_t o = ent * D + c * (D / 4) + t * 8;
        kh[t] = here ? *reinterpret_cast<const uint4*>((const bf16*)sp.khi + o) : make_uint4(0u, 0u, 0u, 0u);
        kl[t] = here ? *reinterpret_cast<const uint4*>((const bf16*)sp.klo + o) : make_uint4(0u, 0u, 0u, 0u);
      }
      const float be = here ? sp.beta[ent] : -INFINITY;
      for (int o = o0; o < o1; o += 16) {
        const int cnt = min(16, o1 - o);
        float s[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (8 * h < cnt) {
            const bf16* qr = q_s + (list[o + min(8 * h + n, cnt - 1)] >> 16) * LD + c * (D / 4);
#pragma unroll
            for (int t = 0; t < KS / 2; ++t) {
              const uint4 x = *reinterpret_cast<const uint4*>(qr + 8 * t);
              nb_mma(s[h], kh[t].x, kl[t].x, kh[t].y, kl[t].y, x.x, x.y);
              nb_mma(s[h], kh[t].z, kl[t].z, kh[t].w, kl[t].w, x.z, x.w);
            }
          }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {                                // pairs 2c, 2c + 1, 8 + 2c, 9 + 2c with block n
          const int h = 8 * (k >> 1) + 2 * c + (k & 1);
          if (h < cnt) {
            const uint32_t le = list[o + h];
            if (n < nb_s[le >> 16] && be != -INFINITY)
              lg_s[(le & 0xffffu) * G + n] = dm.sigma * (s[k >> 1][k & 1] + s[k >> 1][2 + (k & 1)]) + be;
          }
        }
      }
    }
    __syncthreads();

    // ---- step 2: the k2 best blocks of a pair: largest logit first, ties to the lower block; fewer candidates -> all of them
    for (int e = tid; e < nq * m; e += kThreads) {
      const int r = e / m, s = e - r * m, t = row_s[r], j = sel_s[e];
      if (t < 0) continue;
      const size_t pr = ((size_t)pq * dm.N + t) * m + s;
      int32_t* bo = bsel_out + pr * k2;
      bool first = j != 0xffff;                                      // a cluster named twice counts once
      for (int x = 0; first && x < s; ++x) first = sel_s[e - s + x] != j;
      float4* lw = reinterpret_cast<float4*>(lg_s + e * G);
      const float4 la = lw[0], lb = lw[1];
      float lg[G] = {la.x, la.y, la.z, la.w, lb.x, lb.y, lb.z, lb.w};
      uint32_t chosen = first ? 0u : 0xffu;
      if (first && bsel_in != nullptr) {
        for (int x = 0; x < k2; ++x) {
          const int bb = bsel_in[pr * k2 + x];
          const bool take = bb >= 0 && bb < nb_s[r] && !((chosen >> bb) & 1u);   // a block named twice is retrieved once
          if (take) chosen |= 1u << bb;
          bo[x] = take ? bb : -1;
        }
      } else {
        for (int x = 0; x < k2; ++x) {
          float bv = -INFINITY;
          int bi = -1;
#pragma unroll
          for (int bp = 0; bp < G; ++bp)
            if (!((chosen >> bp) & 1u) && lg[bp] > bv) { bv = lg[bp]; bi = bp; }
          bo[x] = bi;
          if (bi >= 0) chosen |= 1u << bi;
        }
      }
      // every other non-empty earlier block of the cluster is a stand-in key of this query
#pragma unroll
      for (int bp = 0; bp < G; ++bp)
        if ((chosen >> bp) & 1u) lg[bp] = -INFINITY;
      lw[0] = make_float4(lg[0], lg[1], lg[2], lg[3]);
      lw[1] = make_float4(lg[4], lg[5], lg[6], lg[7]);
    }
    __syncthreads();

    // ---- step 3
    for (int r = warp; r < nq; r += kWarps) {
      const int t = row_s[r];
      if (t < 0) continue;                                           // (warp-uniform)
      float* lg = lg_s + r * m * G;
      float M = -INFINITY, sum = 0.f;
      for (int e = lane; e < m * G; e += 32) M = fmaxf(M, lg[e]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
      float acc[EPL];
#pragma unroll
      for (int e = 0; e < EPL; ++e) acc[e] = 0.f;
      if (M != -INFINITY) {
        for (int e = lane; e < m * G; e += 32) {
          const float v = lg[e], p = v == -INFINITY ? 0.f : __expf(v - M);
          lg[e] = p;
          sum += p;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        __syncwarp();
        for (int s = 0; s < m; ++s) {
          const int j = sel_s[r * m + s];
          if (j == 0xffff) continue;
          const float4 pa = *reinterpret_cast<const float4*>(lg + s * G), pb = *reinterpret_cast<const float4*>(lg + s * G + 4);
          const float p[G] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w};
          const bf16* nu = (const bf16*)sp.nu + (ebase + j) * D + lane * EPL;
#pragma unroll
          for (int bp = 0; bp < G; ++bp)
            if (p[bp] > 0.f) {                                       // (warp-uniform)
              float nv[EPL];
              ldv<EPL>(nu + (size_t)bp * estep * D, nv);
#pragma unroll
              for (int e = 0; e < EPL; ++e) acc[e] = fmaf(p[bp], nv[e], acc[e]);
            }
        }
        const float inv = 1.f / sum;
#pragma unroll
        for (int e = 0; e < EPL; ++e) acc[e] *= inv;
      }
      const size_t orow = (size_t)pq * dm.N + t;
      stv<EPL>(o_near + orow * D + lane * EPL, acc);
      if (lane == 0) lse_near[orow] = M != -INFINITY ? M + __logf(sum) : -INFINITY;
    }
    __syncthreads();                                                 // the chunk's shared arrays are reused by the next chunk
  }
}

template <int D>
static int block_select_q_d(const Dims& d, const void* Q, const int32_t* off_q, const int32_t* perm_q, const int32_t* sel, const SummPtrs& sp,
                            const int32_t* bsel_in, int32_t* bsel_out, float* o_near, float* lse_near, cudaStream_t st) {
  typedef BqLay<D> L;
  const int smem = L::oOff + d.Ck * 4;
  MUSE_CUDA_OK(cudaFuncSetAttribute(k_block_select_q<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  // a cluster's chunks are shared by several CTAs where one per (cluster, head) would leave SMs idle
  const int per = d.Cq * d.B * d.Hq, chunk = std::min(L::kQ, kNbPairs / d.m);
  const int share = std::max(1, std::min((4 * sm_count() + per - 1) / per, (d.N / d.Cq + chunk - 1) / chunk));
  prof_mark("k_block_select_q", st);
  MUSE_RC(launch_pdl(k_block_select_q<D>, dim3(d.Cq, d.B * d.Hq, share), L::kThreads, smem, st, d, (const bf16*)Q, off_q, perm_q, sel, sp, bsel_in, bsel_out, o_near, lse_near));
  MUSE_LAUNCH_OK();
  return MUSE_OK;
}

int block_select_q(const Dims& d, const void* Q, const int32_t* off_q, const int32_t* perm_q, const int32_t* sel, const SummPtrs& sp,
                   const int32_t* bsel_in, int32_t* bsel_out, float* o_near, float* lse_near, cudaStream_t st) {
  return d.D == 128 ? block_select_q_d<128>(d, Q, off_q, perm_q, sel, sp, bsel_in, bsel_out, o_near, lse_near, st)
                    : block_select_q_d<64>(d, Q, off_q, perm_q, sel, sp, bsel_in, bsel_out, o_near, lse_near, st);
}

}  // namespace muse
