// Backward of the near field of the two-level retrieval (Section "Two-Level Retrieval", second level; Section
// "Output merging", component 2; gradients with the chosen clusters and blocks held constant, Appendix "Centroid
// Gradient Flow").  A stand-in key (i, j, b') - the per-block summary of a non-retrieved earlier block b' of a
// selected cluster j, seen by a query t of query cluster i - has
//     logit = sigma q . kappa + beta,  beta = mu - sigma qbar_i . kappa,   value nu            (kappa, mu, nu of (i, j, b'))
// With L the merged log-sum-exp and delta = dO . O of the query:
//     p = exp(logit - L),  g = p (dO . nu - delta),
//     dq += g sigma kappa,   d nu += p dO,   d kappa += g sigma (q - qbar_i),   d mu += g.
// The sums over queries of d nu, d kappa and of the scalar dS = d mu - d kappa . kappa - d nu . nu (the form in which
// the key-side pass takes the log-mass gradient) are the gradients of the per-block summaries, which that pass then
// carries to the keys and values of bucket (j, b').
//
// Organisation.  A CTA takes the queries of one cluster i over all blocks, up to 256 at a time (bf16 rows in shared memory),
// and lists their (query, slot) pairs by selected cluster j.  Then
//   1. a warp takes a cluster j and the next 16 pairs of its list against the rows of 8 earlier blocks, which it keeps in
//      registers:  S^T = kappa q^T with kappa_hi on rows 0-7 of the product and kappa_lo on rows 8-15, dP^T = nu dO^T;
//      the lanes turn them into p and g in place, where they are B operands (as bf16 high and low parts) of
//      d kappa^T += q^T g,  d nu^T += dO^T p;  the sums over the list go to global memory once, by reductions;
//   2. after a barrier a warp takes a query, lanes sharing D, and adds up g kappa over its pairs in a fixed order.
// The products are 8 blocks by 16 gathered pairs, so they are warp-level mma.sync: tcgen05 products have at least 64 rows.
// Of the pairs of 32 queries of one segment only two or three name the same cluster: a lane per query in step 1 left nine
// lanes in ten idle, and the sums went out after two or three pairs.
//
// Bound: L2 - step 2 reads 256 bytes (D = 64) per pair and block, and the sums leave as 4-byte reductions.  8 heads of two
// sequences of 64k tokens, D = 64, 128 x 128 clusters, 8 slots, 8 blocks: 23.19 ms for a warp per pair with shared-memory
// atomics, 9.88 ms for a lane per query over 32 queries of a segment, 2.68 ms here.
#include <algorithm>
#include "common.cuh"
#include "near.cuh"

namespace muse {

typedef __nv_bfloat16 bf16;

// D = 128 needs 255 registers a thread for its sums
template <int D> struct NbLay {
  static constexpr int kThreads = D == 128 ? 256 : 512, kQ = D == 128 ? 128 : 256;       // queries of a chunk at most
  static constexpr int LD = D + 8;                          // bf16 per query row: ldmatrix rows do not conflict
  static constexpr int oQ = 0, oDO = oQ + kQ * LD * 2, oG = oDO + kQ * LD * 2, oL = oG + kNbPairs * kNbGroup * 4, oDl = oL + kQ * 4, oRow = oDl + kQ * 4,
                       oNb = oRow + kQ * 4, oVis = oNb + kQ * 4, oList = oVis + kNbPairs * 4, oSel = oList + kNbPairs * 4, oQb = oSel + kNbPairs * 2,
                       oOff = oQb + D * 4;                  // then Ck ints
};

__device__ __forceinline__ void nb_ldmatrix_t(uint32_t (&a)[4], const bf16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]) : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
}
// two numbers as packed bf16 high parts and packed bf16 remainders
__device__ __forceinline__ void nb_split(float x, float y, uint32_t& hi, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  const __nv_bfloat162 l = __floats2bfloat162_rn(x - __bfloat162float(h.x), y - __bfloat162float(h.y));
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}

template <int D>
__global__ void __launch_bounds__(NbLay<D>::kThreads, 1)
k_near_bwd(Dims dm, const bf16* __restrict__ Q, const bf16* __restrict__ dO, const float* __restrict__ qbar, const float* __restrict__ LSE,
           const float* __restrict__ delta, const int32_t* __restrict__ off_q, const int32_t* __restrict__ perm_q,
           const int32_t* __restrict__ sel, const int32_t* __restrict__ bsel, SummPtrs sp, float* __restrict__ dQacc,
           float* __restrict__ dkappa_b, float* __restrict__ dnu_b, float* __restrict__ dS_b, int grad_ji) {
  pdl_wait();
  pdl_trigger();
  // grad_ji: the gradient entries are laid out [plane][j][i] (what the tensor-core key-side kernel reads) instead of [plane][i][j]
  typedef NbLay<D> L;
  constexpr int kThreads = L::kThreads, kWarps = kThreads / 32, LD = L::LD, EPL = D / 32, KS = D / 16, G = kNbGroup;
  extern __shared__ __align__(16) unsigned char nb_sm[];
  const int m = dm.m, k2 = dm.k2, SB = dm.SB, Ck = dm.Ck;
  bf16 *q_s = (bf16*)(nb_sm + L::oQ), *do_s = (bf16*)(nb_sm + L::oDO);
  float *g_s = (float*)(nb_sm + L::oG), *L_s = (float*)(nb_sm + L::oL), *dl_s = (float*)(nb_sm + L::oDl), *qb_s = (float*)(nb_sm + L::oQb);
  int *row_s = (int*)(nb_sm + L::oRow), *nb_s = (int*)(nb_sm + L::oNb), *off = (int*)(nb_sm + L::oOff);
  uint32_t *vis_s = (uint32_t*)(nb_sm + L::oVis), *list = (uint32_t*)(nb_sm + L::oList);       // list: query << 16 | pair
  uint16_t* sel_s = (uint16_t*)(nb_sm + L::oSel);
  __shared__ int pre_s[33], p0_s[33], next_s;                        // queries of the cluster before block b + 1; where block b + 1's start
  const int i = blockIdx.x, pq = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, n = lane >> 2, c = lane & 3;
  const int32_t* pm = perm_q + (size_t)pq * dm.N;
  const size_t estep = (size_t)dm.Cq * Ck;
  const size_t ebase = ((size_t)pq * SB * dm.Cq + i) * Ck;           // entry (block 0, i, cluster 0)
  if (warp == 0) {                                                   // SB <= 32
    const int32_t* oq = off_q + (size_t)pq * (dm.S * dm.Cq + 1) + (size_t)(lane + 1) * dm.Cq + i;
    const int p0 = lane < SB ? oq[0] : 0, len = lane < SB ? oq[1] - p0 : 0;
    int pre = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, pre, o); if (lane >= o) pre += v; }
    p0_s[lane] = p0;
    pre_s[lane + 1] = pre;
    if (lane == 0) pre_s[0] = 0;
  }
  for (int d = tid; d < D; d += kThreads) qb_s[d] = qbar[((size_t)pq * dm.Cq + i) * D + d];
  __syncthreads();
  const int total = pre_s[SB], QC = min(L::kQ, kNbPairs / m);
  for (int c0 = blockIdx.z * QC; c0 < total; c0 += gridDim.z * QC) {
    const int nq = min(QC, total - c0);
    // ---- the chunk's queries, their pairs, the list of pairs by selected cluster
    for (int r = tid; r < nq; r += kThreads) {
      int b = 0;
      while (pre_s[b + 1] <= c0 + r) ++b;
      int t = pm[p0_s[b] + c0 + r - pre_s[b]];
      if (!MUSE_IN_RANGE(t, dm.N)) t = -1;
      row_s[r] = t;
      nb_s[r] = b + 1;
      L_s[r] = t >= 0 ? LSE[(size_t)pq * dm.N + t] : 0.f;
      dl_s[r] = t >= 0 ? delta[(size_t)pq * dm.N + t] : 0.f;
    }
    for (int j = tid; j < Ck; j += kThreads) off[j] = 0;
    __syncthreads();
    constexpr int kP = D / 8;                                        // 16-byte pieces of a row
    for (int e = tid; e < nq * 2 * kP; e += kThreads) {
      const int r = e / (2 * kP), w = e / kP % 2, p = e % kP;
      const size_t o = ((size_t)pq * dm.N + max(row_s[r], 0)) * D + p * 8;
      nb_cp_async16((w ? do_s : q_s) + r * LD + p * 8, (w ? dO : Q) + o);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    for (int e = tid; e < nq * m; e += kThreads) {
      const int r = e / m, t = row_s[r], nb = nb_s[r];
      int j = -1;
      uint32_t vis = 0u;                                             // the earlier blocks that stand in for this pair's keys:
      if (t >= 0) {
        const size_t pr = ((size_t)pq * dm.N + t) * m + (e - r * m);
        j = sel[pr];
        if (j < 0 || j >= Ck) j = -1;
        vis = 0xffffffffu >> (32 - nb);
        for (int x = 0; x < k2; ++x) {
          const int bb = bsel[pr * k2 + x];
          if (bb >= 0 && bb < nb) vis &= ~(1u << bb);                // all but those retrieved exactly
        }
      }
      if (vis == 0u) j = -1;
      vis_s[e] = vis;
      sel_s[e] = (uint16_t)(j < 0 ? 0xffff : j);
      if (j >= 0) atomicAdd(&off[j], 1);
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
    for (int g0 = 0; g0 < nbmax; g0 += G) {
      if (tid == 0) next_s = 0;
      __syncthreads();
      for (;;) {
        int j = 0;
        if (lane == 0) j = atomicAdd(&next_s, 1);
        j = __shfl_sync(0xffffffffu, j, 0);
        if (j >= Ck) break;
        const int o0 = j > 0 ? off[j - 1] : 0, o1 = off[j];
        if (o0 == o1) continue;
        // ---- step 1.  Lane (n, c) holds block n's dims c D/4 .. of kappa and nu: the k index of a product is a permutation of D,
        // the same for both operands, so that a lane's operands are 16-byte loads.
        const size_t ent = ebase + (size_t)(g0 + n) * estep + j;
        uint4 kh[KS / 2], kl[KS / 2], nv[KS / 2];
        const bool here = g0 + n < nbmax;
#pragma unroll
        for (int t = 0; t < KS / 2; ++t) {
          const size_t o = ent * D + c * (D / 4) + t * 8;
          kh[t] = here ? *reinterpret_cast<const uint4*>((const bf16*)sp.khi + o) : make_uint4(0u, 0u, 0u, 0u);
          kl[t] = here ? *reinterpret_cast<const uint4*>((const bf16*)sp.klo + o) : make_uint4(0u, 0u, 0u, 0u);
          nv[t] = here ? *reinterpret_cast<const uint4*>((const bf16*)sp.nu + o) : make_uint4(0u, 0u, 0u, 0u);
        }
        const float be = here ? sp.beta[ent] : -INFINITY;
        const bool live = be != -INFINITY;
        float s3 = 0.f;                                              // sigma qbar_i . kappa of block n
#pragma unroll
        for (int t = 0; t < KS / 2; ++t) {
          const uint32_t h[4] = {kh[t].x, kh[t].y, kh[t].z, kh[t].w}, l[4] = {kl[t].x, kl[t].y, kl[t].z, kl[t].w};
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            const float2 qv = *reinterpret_cast<const float2*>(qb_s + c * (D / 4) + t * 8 + 2 * x);
            s3 = fmaf(qv.x, __uint_as_float(h[x] << 16) + __uint_as_float(l[x] << 16), s3);
            s3 = fmaf(qv.y, __uint_as_float(h[x] & 0xffff0000u) + __uint_as_float(l[x] & 0xffff0000u), s3);
          }
        }
        s3 += __shfl_xor_sync(0xffffffffu, s3, 1);
        s3 += __shfl_xor_sync(0xffffffffu, s3, 2);
        s3 *= dm.sigma;
        float aka[KS][4], anu[KS][4], ds = 0.f, gsum = 0.f;          // sums over the list: [dims of tile: n, n + 8][blocks 2c, 2c + 1]
        uint32_t seen = 0u;
#pragma unroll
        for (int t = 0; t < KS; ++t)
#pragma unroll
          for (int x = 0; x < 4; ++x) { aka[t][x] = 0.f; anu[t][x] = 0.f; }
        for (int o = o0; o < o1; o += 16) {
          const int cnt = min(16, o1 - o);
          float s[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}}, dp[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (8 * h < cnt) {
              const int r = list[o + min(8 * h + n, cnt - 1)] >> 16;
              const bf16 *qr = q_s + r * LD + c * (D / 4), *gr = do_s + r * LD + c * (D / 4);
#pragma unroll
              for (int t = 0; t < KS / 2; ++t) {
                const uint4 x = *reinterpret_cast<const uint4*>(qr + 8 * t), y = *reinterpret_cast<const uint4*>(gr + 8 * t);
                nb_mma(s[h], kh[t].x, kl[t].x, kh[t].y, kl[t].y, x.x, x.y);
                nb_mma(s[h], kh[t].z, kl[t].z, kh[t].w, kl[t].w, x.z, x.w);
                nb_mma(dp[h], nv[t].x, 0u, nv[t].y, 0u, y.x, y.y);
                nb_mma(dp[h], nv[t].z, 0u, nv[t].w, 0u, y.z, y.w);
              }
            }
          }
          float p[4], g[4];                                          // pairs 2c, 2c + 1, 8 + 2c, 9 + 2c with block n
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int h = 8 * (k >> 1) + 2 * c + (k & 1);
            p[k] = g[k] = 0.f;
            if (h < cnt) {
              const uint32_t le = list[o + h];
              const int r = le >> 16, e = le & 0xffffu;
              const uint32_t vis = vis_s[e];
              const float lg = dm.sigma * (s[k >> 1][k & 1] + s[k >> 1][2 + (k & 1)]), dv = dp[k >> 1][k & 1];
              if (live && ((vis >> (g0 + n)) & 1u)) {
                p[k] = __expf(lg + be - L_s[r]);
                g[k] = p[k] * (dv - dl_s[r]);
                // the scalar the key-side pass wants per entry: d mu - d kappa . kappa - d nu . nu
                ds += g[k] * (1.f - (lg - s3)) - p[k] * dv;
                gsum += g[k];
                seen = 1u;
              }
              g_s[e * G + n] = g[k];
            }
          }
          uint32_t gh[2], gl[2], ph[2], pl[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) { nb_split(g[2 * h], g[2 * h + 1], gh[h], gl[h]); nb_split(p[2 * h], p[2 * h + 1], ph[h], pl[h]); }
          const int ro = (list[o + min((lane & 7) + ((lane >> 4) << 3), cnt - 1)] >> 16) * LD + ((lane >> 3) & 1) * 8;
#pragma unroll
          for (int t = 0; t < KS; ++t) {
            uint32_t a[4];
            nb_ldmatrix_t(a, q_s + ro + 16 * t);
            nb_mma(aka[t], a[0], a[1], a[2], a[3], gh[0], gh[1]);
            nb_mma(aka[t], a[0], a[1], a[2], a[3], gl[0], gl[1]);
            nb_ldmatrix_t(a, do_s + ro + 16 * t);
            nb_mma(anu[t], a[0], a[1], a[2], a[3], ph[0], ph[1]);
            nb_mma(anu[t], a[0], a[1], a[2], a[3], pl[0], pl[1]);
          }
        }
        ds += __shfl_xor_sync(0xffffffffu, ds, 1);
        gsum += __shfl_xor_sync(0xffffffffu, gsum, 1);
        ds += __shfl_xor_sync(0xffffffffu, ds, 2);
        gsum += __shfl_xor_sync(0xffffffffu, gsum, 2);
        const uint32_t any = __ballot_sync(0xffffffffu, seen != 0u); // blocks without a stand-in of this list have nothing to add
        const auto entry = [&](int bp) {
          return grad_ji ? (((size_t)pq * SB + g0 + bp) * Ck + j) * dm.Cq + i : ebase + (size_t)(g0 + bp) * estep + j;
        };
        if (c == 0 && ((any >> (4 * n)) & 15u) != 0u) atomicAdd(dS_b + entry(n), ds);
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const int bp = 2 * c + x;
          const float gs = __shfl_sync(0xffffffffu, gsum, 4 * bp);
          if (((any >> (4 * bp)) & 15u) == 0u) continue;
          float *ka = dkappa_b + entry(bp) * D, *nu = dnu_b + entry(bp) * D;
#pragma unroll
          for (int t = 0; t < KS; ++t) {
            const int d = 16 * t + n;
            atomicAdd(ka + d, dm.sigma * (aka[t][x] - gs * qb_s[d]));
            atomicAdd(ka + d + 8, dm.sigma * (aka[t][2 + x] - gs * qb_s[d + 8]));
            atomicAdd(nu + d, anu[t][x]);
            atomicAdd(nu + d + 8, anu[t][2 + x]);
          }
        }
      }
      __syncthreads();
      // ---- step 2: a warp per query, lanes share D: sum of g kappa (the far-field and local parts are already in the accumulator)
      for (int r = warp; r < nq; r += kWarps) {
        if (row_s[r] < 0) continue;                                  // (warp-uniform)
        float acc[EPL];
#pragma unroll
        for (int e = 0; e < EPL; ++e) acc[e] = 0.f;
        for (int s = 0; s < m; ++s) {
          const int j = sel_s[r * m + s];
          if (j == 0xffff) continue;
          const float4 ga = *reinterpret_cast<const float4*>(g_s + (r * m + s) * G), gb = *reinterpret_cast<const float4*>(g_s + (r * m + s) * G + 4);
          const float g[G] = {ga.x, ga.y, ga.z, ga.w, gb.x, gb.y, gb.z, gb.w};
          const size_t o = (ebase + (size_t)g0 * estep + j) * D + lane * EPL;
#pragma unroll
          for (int bp = 0; bp < G; ++bp)
            if (g[bp] != 0.f) {
              float kh[EPL], kl[EPL];
              ldv<EPL>((const bf16*)sp.khi + o + (size_t)bp * estep * D, kh);
              ldv<EPL>((const bf16*)sp.klo + o + (size_t)bp * estep * D, kl);
#pragma unroll
              for (int e = 0; e < EPL; ++e) acc[e] = fmaf(g[bp], kh[e] + kl[e], acc[e]);
            }
        }
        float* dst = dQacc + ((size_t)pq * dm.N + row_s[r]) * D + lane * EPL;
        float cur[EPL];
        ldv<EPL>(dst, cur);
#pragma unroll
        for (int e = 0; e < EPL; ++e) cur[e] = fmaf(dm.sigma, acc[e], cur[e]);
        stv<EPL>(dst, cur);
      }
      __syncthreads();                                               // g_s and the lists are refilled
    }
  }
}

// fp32 gradient rows -> bf16 (the operand type of the tensor-core key-side kernel), same layout
__global__ void k_grad_to_bf16(const float* __restrict__ in, long long n4, __nv_bfloat16* __restrict__ out) {
  pdl_wait();
  pdl_trigger();
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n4) return;
  st4(out + 4 * e, ld4(in + 4 * e));
}

int grad_to_bf16(const float* in, size_t n, void* out, cudaStream_t st) {
  const long long n4 = (long long)(n / 4);
  prof_mark("k_grad_to_bf16", st);
  MUSE_RC(launch_pdl(k_grad_to_bf16, dim3((unsigned)((n4 + 255) / 256)), 256, 0, st, in, n4, (__nv_bfloat16*)out));
  MUSE_LAUNCH_OK();
  return MUSE_OK;
}

template <int D>
static int near_bwd_d(const Dims& d, const void* Q, const void* dO, const float* qbar, const float* LSE, const float* delta, const int32_t* off_q,
                      const int32_t* perm_q, const int32_t* sel, const int32_t* bsel, const SummPtrs& sp, float* dQacc, float* dkappa_b,
                      float* dnu_b, float* dS_b, int grad_ji, cudaStream_t st) {
  typedef NbLay<D> L;
  const int smem = L::oOff + d.Ck * 4;                       // Ck <= 4096: at most 180 KB
  MUSE_CUDA_OK(cudaFuncSetAttribute(k_near_bwd<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  // a cluster's chunks are shared by several CTAs where one per (cluster, head) would leave SMs idle
  const int per = d.Cq * d.B * d.Hq, chunk = std::min(L::kQ, kNbPairs / d.m);
  const int share = std::max(1, std::min((2 * sm_count() + per - 1) / per, (d.N / d.Cq + chunk - 1) / chunk));
  prof_mark("k_near_bwd", st);
  MUSE_RC(launch_pdl(k_near_bwd<D>, dim3(d.Cq, d.B * d.Hq, share), L::kThreads, smem, st, d, (const bf16*)Q, (const bf16*)dO, qbar, LSE, delta, off_q, perm_q, sel, bsel, sp, dQacc, dkappa_b, dnu_b, dS_b, grad_ji));
  MUSE_LAUNCH_OK();
  return MUSE_OK;
}

// k2 > 0 (and with it S > 1 blocks) is built for bf16 only
int near_bwd(const Dims& d, const void* Q, const void* dO, const float* qbar, const float* LSE, const float* delta, const int32_t* off_q,
             const int32_t* perm_q, const int32_t* sel, const int32_t* bsel, const SummPtrs& sp, float* dQacc, float* dkappa_b, float* dnu_b,
             float* dS_b, int grad_ji, cudaStream_t st) {
  return d.D == 128 ? near_bwd_d<128>(d, Q, dO, qbar, LSE, delta, off_q, perm_q, sel, bsel, sp, dQacc, dkappa_b, dnu_b, dS_b, grad_ji, st)
                    : near_bwd_d<64>(d, Q, dO, qbar, LSE, delta, off_q, perm_q, sel, bsel, sp, dQacc, dkappa_b, dnu_b, dS_b, grad_ji, st);
}

}  // namespace muse
