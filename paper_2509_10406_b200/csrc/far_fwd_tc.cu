// Far-field forward on the tensor cores (bf16 mode, D = 64 or 128, Ck <= 2048).  Clusters come in tiles of 128; the
// tensor maps end at Ck, so the rows of the last tile past it are zeros, and their beta is taken as -infinity.
// One CTA per (query cluster i, plane, head) segment; its queries (32 on average at the headline
// sizes, up to 64 per pass) share the Ck accumulated summaries of (i, plane).  The summaries sit
// on the MMA M side (128 clusters per tile, one TMEM lane each) and the queries on the N side
// (64 columns), so the segment streams its summaries once:
//   A  scores^T[j][r] = (kappa_hi[j] + kappa_lo[j]) . q[r]   two accumulating MMAs per tile,
//      kappa tiles streamed by TMA through a ring that spans the whole operand area;
//      score = sigma * that + beta[j] (Eq. 6).  All 64 x Ck scores stay in TMEM (512 columns).
//   B  16 queries at a time: TMEM -> shared memory transposed to [r][j] fp32
//   C  per query (one warp each): top-m selection, far-set softmax, P written as a bf16 operand; the scores stay in registers from
//      one end to the other (read again for the maximum and the weights: 4800 cycles a step of eight queries, now 2900; the whole
//      kernel 6.25 -> 5.99 ms at 128k tokens, 512 x 2048 clusters, D = 128; 1461 -> 1450 us at 64k, 256 x 1024)
//   D  out^T[d][r] = sum_j nu[j][d] P[r][j]      nu in units of 16 KB (MN-major A operand) streamed by TMA through the score rows and,
//      as it is used up, P (through the score rows alone, 64 KB, 27 bytes a clock: 5.99 -> 5.75 ms, 1450 -> 1429 us)
//      (bringing them, or the next segment's kappa, into L2 while phase C runs evicts what others are about to read:
//      6.25 ms without, 6.56 with nu, 6.9 to 8.4 with kappa at 128k tokens, 512 x 2048 clusters, D = 128)
//   E  TMEM -> o_far (thread = d, coalesced over d for each query)
#include <cuda.h>
#include "common.cuh"
#include "tc05.cuh"

namespace muse {

typedef __nv_bfloat16 bf16;
int make_tmap_bf16_nd(void* out_map, const void* base, int rank, const uint64_t* dims, const uint64_t* strides_bytes, const uint32_t* box);

constexpr int kFJ = 128;                            // clusters per tile
// Queries per pass FR and per selection step FQ (one warp each) are template parameters: 64 / 16 up to 1024
// key clusters, 32 / 8 up to 2048 (all FR x Ck scores of a pass live in the 512 TMEM columns, P and the score
// rows of a step in shared memory).
constexpr int kMaxStA = 6;
constexpr int kSlot = 16 * 1024, kMaxUnits = 32;    // phase D: nu comes in units of 16 KB (64 clusters at D = 128, 128 at D = 64)
constexpr int kCandMax = 128;                       // candidates kept by the compacting selection (4 per lane)

struct FarBars { uint64_t fullA[kMaxStA], emptyA[kMaxStA], fullD[kMaxUnits], emptyD[kMaxUnits], done; };


// Scores of a lane: fours of consecutive clusters, 128 apart; v[k] is cluster 4 lane + 128 (k / 4) + k % 4.  (16-byte reads of a
// score row without bank conflicts, and eight bytes of P at a time.)
__device__ __forceinline__ int cluster_of(int lane, int k) { return 4 * lane + 128 * (k >> 2) + (k & 3); }
template <int NKMAX>
__device__ __forceinline__ void load_scores(const float* s, int NK, int lane, float (&v)[NKMAX]) {
#pragma unroll
  for (int k = 0; k < NKMAX; k += 4) {
    float4 x = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    if (k < NK) x = *reinterpret_cast<const float4*>(s + 4 * lane + 32 * k);
    v[k] = x.x; v[k + 1] = x.y; v[k + 2] = x.z; v[k + 3] = x.w;
  }
}

// Top-m of one query's scores s[0..Ck) (one warp; Ck <= 32 NKMAX), which the lanes hold in v.  Writes the chosen clusters to
// so[0..m) (-1 padded, in no particular order), and removes them from the far set by setting
// their score to -inf, in v at least.  Scores become order-preserving integer keys; everything above the key T
// of the m-th largest is taken and, among ties at T, the lowest cluster indices.
//
// Fast path (m <= 64, `may_compact`): the m-th largest of the 64 per-lane top-two keys, found by a
// bitonic sort across the warp (two keys per lane, shuffles only), bounds the m-th largest score
// from below, and on random data only about m + 4 scores reach it.  Those candidates are
// compacted into `cand` (kCandMax keys then kCandMax indices, 128-byte segments `seg` bytes apart;
// a lane-prefix sum gives every lane its slots, so the scatter needs no votes) and T is the largest key that m candidates reach: a
// lane counts for its two (bisection over 4 keys per lane, 20 dependent reductions, where there are more than 64).  The code is laid
// out for instruction-level parallelism: a warp's chain of dependent votes and reductions, not the issue rate, bounds the selection.
// General path (any m, many equal scores, fewer than m finite scores): bisection over all keys.
template <int NKMAX>
__device__ __forceinline__ void select_top_m(float* s, int Ck, int m, int32_t* so, int lane, unsigned char* cand, int seg,
                                             bool may_compact, float (&v)[NKMAX]) {
  const int NK = Ck >> 5;                       // scores per lane (<= NKMAX)
  auto to_key = [](float x) {
    const uint32_t b = __float_as_uint(x);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
  };
  const uint32_t kFinite = 0x00800000u;         // smallest key above key(-inf) = 0x007fffff
  const uint32_t lt = (1u << lane) - 1u;
  float f1 = -INFINITY, f2 = -INFINITY;         // the lane's largest and second largest score
#pragma unroll
  for (int k = 0; k < NKMAX; ++k) {
    f2 = fmaxf(f2, fminf(f1, v[k]));
    f1 = fmaxf(f1, v[k]);
  }
  const uint32_t m1 = to_key(f1), m2 = to_key(f2);
  if (may_compact && m >= 1 && m <= 64) {
    // bitonic sort, descending, of the 64 keys e = 2 lane + r held as (v0, v1)
    uint32_t v0 = m1, v1 = m2;
    const int e2 = lane << 1;
#pragma unroll
    for (int k = 2; k <= 64; k <<= 1) {
      const bool desc = (e2 & k) == 0;
#pragma unroll
      for (int j = k >> 1; j >= 2; j >>= 1) {
        const uint32_t p0 = __shfl_xor_sync(0xffffffffu, v0, j >> 1), p1 = __shfl_xor_sync(0xffffffffu, v1, j >> 1);
        const bool keep_max = ((e2 & j) == 0) == desc;
        v0 = keep_max ? max(v0, p0) : min(v0, p0);
        v1 = keep_max ? max(v1, p1) : min(v1, p1);
      }
      const uint32_t hi = max(v0, v1), lo = min(v0, v1);
      v0 = desc ? hi : lo;
      v1 = desc ? lo : hi;
    }
    const uint32_t lb = __shfl_sync(0xffffffffu, ((m - 1) & 1) ? v1 : v0, (m - 1) >> 1);
    const uint32_t kmx = __shfl_sync(0xffffffffu, v0, 0);
    uint32_t msk[(NKMAX + 31) / 32] = {};                     // this lane's candidates, one bit per score
    // (float comparison: the same set as by key, plus -0 beside +0, which does no harm)
    const uint32_t lbb = (lb & 0x80000000u) ? (lb & 0x7fffffffu) : ~lb;
    const float lbf = __uint_as_float(lbb);
#pragma unroll
    for (int k = 0; k < NKMAX; ++k) msk[k >> 5] |= v[k] >= lbf ? 1u << (k & 31) : 0u;
    int cl = 0;
#pragma unroll
    for (int w = 0; w < (NKMAX + 31) / 32; ++w) cl += __popc(msk[w]);
    int incl = cl;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += t;
    }
    const int ncand = __shfl_sync(0xffffffffu, incl, 31);
    if (lb >= kFinite && ncand <= kCandMax) {
      // a lane holds one or two candidates as a rule: walk its mask and fetch the scores again
      int pos = incl - cl;
#pragma unroll
      for (int w = 0; w < (NKMAX + 31) / 32; ++w) {
        for (uint32_t mm = msk[w]; mm != 0u; mm &= mm - 1u, ++pos) {
          const int j = cluster_of(lane, 32 * w + __ffs((int)mm) - 1);
          *reinterpret_cast<uint32_t*>(cand + (pos >> 5) * seg + (pos & 31) * 4) = to_key(s[j]);
          *reinterpret_cast<int32_t*>(cand + (4 + (pos >> 5)) * seg + (pos & 31) * 4) = j;
        }
      }
      __syncwarp();
      uint32_t ck[4];
      int32_t ci[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const bool in = lane + 32 * q < ncand;
        ck[q] = in ? *reinterpret_cast<const uint32_t*>(cand + q * seg + lane * 4) : 0u;
        ci[q] = in ? *reinterpret_cast<const int32_t*>(cand + (4 + q) * seg + lane * 4) : 0x7fffffff;
      }
      auto count4 = [&](uint32_t thr) {
        return (int)__reduce_add_sync(0xffffffffu, (unsigned)((ck[0] >= thr) + (ck[1] >= thr) + (ck[2] >= thr) + (ck[3] >= thr)));
      };
      uint32_t T;
      if (ncand <= 64) {
        int c0 = 0, c1 = 0;                                     // candidates that reach this lane's two
        for (int q = 0; q < ncand; q += 4) {
          const uint4 x = *reinterpret_cast<const uint4*>(cand + (q >> 5) * seg + (q & 31) * 4);       // (past ncand: what was there before)
          c0 += (x.x >= ck[0]) + (q + 1 < ncand && x.y >= ck[0]) + (q + 2 < ncand && x.z >= ck[0]) + (q + 3 < ncand && x.w >= ck[0]);
          c1 += (x.x >= ck[1]) + (q + 1 < ncand && x.y >= ck[1]) + (q + 2 < ncand && x.z >= ck[1]) + (q + 3 < ncand && x.w >= ck[1]);
        }
        T = __reduce_max_sync(0xffffffffu, max(c0 >= m ? ck[0] : 0u, c1 >= m ? ck[1] : 0u));
      } else {
        const int shared = __clz((int)(kmx ^ lb));              // 32 if the interval is a single key
        T = shared >= 32 ? kmx : (kmx & ~(0xffffffffu >> shared));
        for (int bit = 31 - shared; bit >= 0; --bit) {
          const uint32_t c2 = T | (1u << bit);
          const int c = count4(c2);
          if (c >= m) { T = c2; if (c == m) break; }
        }
      }
      const int places = m - count4(T + 1u);                    // ties at T to take (>= 0)
      int need = places;
      const int ntie = (int)__reduce_add_sync(0xffffffffu, (unsigned)((ck[0] == T) + (ck[1] == T) + (ck[2] == T) + (ck[3] == T)));
      bool take[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) take[q] = ck[q] > T || (ntie <= need && ck[q] == T);
      if (ntie > need) {
        // more ties than places: lowest cluster indices first
        for (; need > 0; --need) {
          int jm = 0x7fffffff;
#pragma unroll
          for (int q = 0; q < 4; ++q) jm = min(jm, (ck[q] == T && !take[q]) ? ci[q] : 0x7fffffff);
          jm = __reduce_min_sync(0xffffffffu, jm);
#pragma unroll
          for (int q = 0; q < 4; ++q) take[q] = take[q] || (ck[q] == T && ci[q] == jm);
        }
      }
      // T as a number tells the taken ones, but where some of its ties are not, or where it is a zero (-0 has a key of its own)
      const float Tf = __uint_as_float((T & 0x80000000u) ? (T & 0x7fffffffu) : ~T);
      const bool mark = ntie > places || Tf == 0.f;
      int base = 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (32 * q < ncand) {
          const uint32_t ms = __ballot_sync(0xffffffffu, take[q]);
          if (take[q]) { so[base + __popc(ms & lt)] = ci[q]; if (mark) s[ci[q]] = -INFINITY; }
          base += __popc(ms);
        }
      }
      for (int k = base + lane; k < m; k += 32) so[k] = -1;
      if (mark) {
        __syncwarp();
        load_scores<NKMAX>(s, NK, lane, v);
      } else {
#pragma unroll
        for (int k = 0; k < NKMAX; ++k) v[k] = v[k] >= Tf ? -INFINITY : v[k];
      }
      return;
    }
  }

  uint32_t key[NKMAX];                          // here a lane's scores are 32 apart: the order of the votes is that of the clusters
#pragma unroll
  for (int k = 0; k < NKMAX; ++k) key[k] = to_key(k < NK ? s[lane + 32 * k] : -INFINITY);
  auto count_ge = [&](uint32_t thr) {           // lane-local count, then one warp reduction
    int c = 0;
#pragma unroll
    for (int k = 0; k < NKMAX; ++k) c += key[k] >= thr ? 1 : 0;
    return (int)__reduce_add_sync(0xffffffffu, (unsigned)c);
  };
  uint32_t kmn = 0xffffffffu;                   // smallest finite key
  int nfin = 0;
#pragma unroll
  for (int k = 0; k < NKMAX; ++k) {
    const bool fin = key[k] >= kFinite;
    nfin += fin ? 1 : 0;
    kmn = min(kmn, fin ? key[k] : 0xffffffffu);
  }
  const bool take_all = (int)__reduce_add_sync(0xffffffffu, (unsigned)nfin) <= m;
  uint32_t T = kFinite;
  if (!take_all) {
    const uint32_t kmx = __reduce_max_sync(0xffffffffu, m1);
    kmn = __reduce_min_sync(0xffffffffu, kmn);
    const int shared = __clz((int)(kmx ^ kmn));            // 32 if the interval is a single key
    T = shared >= 32 ? kmx : (kmx & ~(0xffffffffu >> shared));
    for (int bit = 31 - shared; bit >= 0; --bit) {
      const uint32_t c2 = T | (1u << bit);
      const int c = count_ge(c2);
      if (c >= m) { T = c2; if (c == m) break; }
    }
  }
  int base = 0, ties_seen = 0;
  const int need = take_all ? 0 : m - count_ge(T + 1u);
#pragma unroll
  for (int k = 0; k < NKMAX; ++k) {
    if (k < NK) {
      const bool tie = !take_all && key[k] == T;
      const bool gt = take_all ? key[k] >= kFinite : key[k] > T;
      const uint32_t mt = __ballot_sync(0xffffffffu, tie);
      const bool take = gt || (tie && ties_seen + __popc(mt & lt) < need);
      ties_seen += __popc(mt);
      const uint32_t ms = __ballot_sync(0xffffffffu, take);
      if (take) { so[base + __popc(ms & lt)] = lane + 32 * k; s[lane + 32 * k] = -INFINITY; }
      base += __popc(ms);
    }
  }
  for (int k = base + lane; k < m; k += 32) so[k] = -1;
  __syncwarp();
  load_scores<NKMAX>(s, NK, lane, v);
}

// NKMAX: scores per lane that the selection keeps in registers (Ck <= 32 NKMAX); MINB: CTAs per SM the register
// budget is set for.  With few key clusters the per-query selection, a chain of dependent warp operations, is what
// takes the time: small instances (few registers, few TMEM columns) put several CTAs on an SM.
template <int FR, int FQ, int D, int NKMAX, int MINB>
__global__ void __launch_bounds__(FQ * 32, MINB)
k_far_fwd_tc(Dims dm, const __grid_constant__ CUtensorMap tm_khi, const __grid_constant__ CUtensorMap tm_klo,
             const __grid_constant__ CUtensorMap tm_nu, const bf16* __restrict__ Q, const int32_t* __restrict__ off_q,
             const int32_t* __restrict__ perm_q, const float* __restrict__ mu, const float* __restrict__ beta,
             const int32_t* __restrict__ sel_in, int32_t* __restrict__ sel_out, float* __restrict__ o_far,
             float* __restrict__ lse_far, int p_bytes, int sc_bytes, int nsA, int tcols, int* __restrict__ status) {
  pdl_wait();
  constexpr int NT = FQ * 32, NTG = FQ / 4, KT = 16 / NTG;   // threads; tile groups in the TMEM read-out; cluster tiles per group
  constexpr int kTileBytes = kFJ * D * 2, G = D / 64;        // one [128 clusters][D] bf16 operand tile; 128-byte column groups of a row
  extern __shared__ __align__(1024) unsigned char sm_raw[];
  __shared__ FarBars bars;
  __shared__ uint32_t tbase_s;
  __shared__ int32_t rows[FR];
  __shared__ float rinv[FR];
  __shared__ int32_t selq[kMaxM];
  // phase D: where unit u of nu goes, and after which unit's products (-1: at once).  The first units go to the score region; a unit's place
  // is free after its own products, and so is the part of P that they have read last: every kPer units' worth of P makes a further place
  constexpr int KU = kSlot / (D * 2), kPer = kSlot / (KU * FR * 2);
  __shared__ int16_t slot_s[kMaxUnits], after_s[kMaxUnits];
  const int i = blockIdx.x, pl = blockIdx.y, pq = blockIdx.z;
  const int blk = dm.causal ? pl + 1 : 0, Ck = dm.Ck, NJ = (Ck + kFJ - 1) / kFJ, CkP = NJ * kFJ, m = dm.m;   // CkP: clusters rounded up to whole tiles
  const int tid = threadIdx.x, warp = tc::warp_index(), lane = tid & 31;
  const int32_t* oq = off_q + (size_t)pq * (dm.S * dm.Cq + 1) + (size_t)blk * dm.Cq + i;
  const int p0 = oq[0], p1 = oq[1];
  if (p0 >= p1) return;
  // operand area: phase A uses all of it as the kappa ring; afterwards P (bf16 [64][Ck]) sits at
  // its start and the score rows of the current 16 queries, later nu, behind it
  unsigned char* sm = sm_raw + ((1024u - (tc::smem_u32(sm_raw) & 1023u)) & 1023u);
  unsigned char* Pm = sm;
  float* sc = reinterpret_cast<float*>(sm + p_bytes);
  unsigned char* Qs = sm + p_bytes + sc_bytes;
  const int seg = (pq * dm.SB + pl) * dm.Cq + i;
  const size_t ent0 = (size_t)seg * Ck;
  const float* mup = mu + ent0;
  const float* bep = beta + ent0;
  const bf16* Qp = Q + (size_t)pq * dm.N * D;
  const int32_t* pm = perm_q + (size_t)pq * dm.N;

  if (warp == 0) tc::tmem_alloc(&tbase_s, tcols);
  if (tid == 0) {
    for (int s = 0; s < kMaxStA; ++s) { tc::mbar_init(&bars.fullA[s], 1); tc::mbar_init(&bars.emptyA[s], 1); }
    for (int s = 0; s < kMaxUnits; ++s) { tc::mbar_init(&bars.fullD[s], 1); tc::mbar_init(&bars.emptyD[s], 1); }
    tc::mbar_init(&bars.done, 1);
    tc::mbar_init_fence();
  }
  if (dm.sel_mode == MUSE_SEL_PER_QCLUSTER && sel_in == nullptr && m > 0 && warp == 1) {
    // one selection per segment: rank clusters by accumulated log-mass alone
    float* tmp = sc;
    for (int j = lane; j < Ck; j += 32) tmp[j] = mup[j];
    __syncwarp();
    for (int k = 0; k < m; ++k) {
      float bv = -INFINITY; int bi = 0x7fffffff;
      for (int j = lane; j < Ck; j += 32) { float v = tmp[j]; if (v > bv) { bv = v; bi = j; } }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        float ov = __shfl_xor_sync(0xffffffffu, bv, o); int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
      }
      if (lane == 0) selq[k] = bv == -INFINITY ? -1 : bi;
      if (bv != -INFINITY && (bi & 31) == lane) tmp[bi] = -INFINITY;
      __syncwarp();
    }
  }
  if (tid == 64) {
    const int n0 = sc_bytes / kSlot, NU = CkP / KU;
    for (int u = 0; u < NU; ++u) {
      const int e = u - n0, g = e / (kPer + 1), r = e % (kPer + 1);            // (of kPer + 1 places in turn the last one is P's)
      slot_s[u] = (int16_t)(e < 0 ? u : r < kPer ? slot_s[g * kPer + r] : n0 + g);
      after_s[u] = (int16_t)(e < 0 ? -1 : g * kPer + min(r, kPer - 1));
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  pdl_trigger();                                           // (tensor memory has been allocated)
  const uint32_t tbase = tbase_s;
  uint32_t cntA = 0, done_ph = 0, phD = 0;   // tiles of the earlier passes (same in every thread); phase of `done`
  bool ok = true;
  // TMA producers: warps 0, 2, 3, 4 (an elected lane each).  One thread sustains only about 30 bytes per clock
  // (every bulk-tensor instruction holds it for some 270 clocks per 16 KB box, every wait after one
  // for some 500), several threads add up.  Producer p serves the tiles whose running index is
  // p modulo the producer count, and that count divides the ring depth, so a ring stage always
  // belongs to one producer and its waits on the stage's barrier never fall a phase behind.
  const int prod = warp == 0 ? 0 : (warp >= 2 && warp <= 4) ? warp - 1 : -1;
  const int WA = nsA % 4 == 0 ? 4 : nsA % 3 == 0 ? 3 : nsA % 2 == 0 ? 2 : 1;
  const int lq = warp & 3, tg = warp >> 2;            // TMEM lane quarter of this warp, tile group

  for (int r0 = p0; r0 < p1 && ok; r0 += FR) {
    const int n = min(FR, p1 - r0);
    // ---- A: scores^T for all clusters, kappa_hi / kappa_lo tiles through an nsA-stage TMA ring;
    //         the producers load (TMA), thread 32 consumes (MMA), so neither waits for the other's latency.
    //         The first ring-full of tiles is requested before the query rows are gathered.
    // (ring stage, phase and owning producer of a tile advance by increments: no division per tile)
    const int sA0 = cntA % nsA, phA0 = (cntA / nsA) & 1;
    int sa = sA0, pha = phA0, wa = sA0 % WA;             // of the next tile this producer looks at
    auto next_a = [&]() {
      if (++sa == nsA) { sa = 0; pha ^= 1; }
      if (++wa == WA) wa = 0;
    };
    auto produce_a = [&](int t) {
      const int s = sa;
      if (!tc::mbar_wait(&bars.emptyA[s], pha ^ 1)) { ok = false; return; }
      tc::mbar_expect_tx_warp(&bars.fullA[s], kTileBytes);
      const void* map = (t & 1) ? (const void*)&tm_klo : (const void*)&tm_khi;
      for (int g = 0; g < G; ++g) tc::tma_load_3d_warp(sm + s * kTileBytes + g * kFJ * 128, map, 64 * g, (t >> 1) * kFJ, seg, &bars.fullA[s]);
    };
    const int TA = 2 * NJ, TA0 = min(nsA, TA);
    if (prod >= 0 && prod < WA)
      for (int t = 0; t < TA0 && ok; ++t, next_a())
        if (wa == prod) produce_a(t);
    if (tid < FR) rows[tid] = tid < n ? pm[r0 + tid] : -1;
    // query rows -> K-major swizzled tile [FR][D] bf16 (G blocks of [FR][128 B])
    // (all of a thread's row numbers, then all of its rows are on their way at once: nothing else hides their latency)
    constexpr int IT = (FR * (D / 8) + NT - 1) / NT;
    int tq[IT];
    uint4 vq[IT];
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const int r = (tid + it * NT) / (D / 8);
      tq[it] = r < n && MUSE_IN_RANGE(r0 + r, dm.N) ? pm[r0 + r] : -1;
      if (tq[it] >= 0 && !MUSE_IN_RANGE(tq[it], dm.N)) tq[it] = -1;
    }
#pragma unroll
    for (int it = 0; it < IT; ++it)
      vq[it] = tq[it] >= 0 ? reinterpret_cast<const uint4*>(Qp + (size_t)tq[it] * D)[(tid + it * NT) % (D / 8)] : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const int r = (tid + it * NT) / (D / 8), ck = (tid + it * NT) % (D / 8);
      if (r < FR) *reinterpret_cast<uint4*>(Qs + (ck >> 3) * FR * 128 + tc::sw128_off(r, ck & 7)) = vq[it];
    }
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    if (prod >= 0) {
      if (prod < WA)
        for (int t = TA0; t < TA && ok; ++t, next_a())
          if (wa == prod) produce_a(t);
    } else if (warp == 1) {
      tc::fence_after_sync();
      const uint32_t idesc = tc::idesc_bf16(kFJ, FR, 0, 0);
      const uint64_t dq0 = tc::smem_desc_sw128(tc::smem_u32(Qs), 16, 1024), da0 = tc::smem_desc_sw128(tc::smem_u32(sm), 16, 1024);
      const int T = 2 * NJ;
      for (int u = 0, s = sA0, ph = phA0; u < T; ++u) {
        if (!tc::mbar_wait(&bars.fullA[s], ph)) { ok = false; break; }
        const uint64_t da = tc::desc_step(da0, (uint32_t)s * kTileBytes);
        const uint32_t dcol = tbase + (u >> 1) * FR;

#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks)
          tc::mma_bf16_ss_warp(dcol, tc::desc_step(da, (ks / 4) * kFJ * 128 + (ks % 4) * 32),
                          tc::desc_step(dq0, (ks / 4) * FR * 128 + (ks % 4) * 32), idesc, (u & 1) || ks > 0);
        tc::mma_commit_warp(&bars.emptyA[s]);
        if (++s == nsA) { s = 0; ph ^= 1; }
      }
      if (ok) tc::mma_commit_warp(&bars.done);
    }
    float bq[KT];                                       // beta of this thread's clusters, loaded ahead of the TMEM reads
#pragma unroll
    for (int k = 0; k < KT; ++k) { const int j = (tg + NTG * k) * kFJ + (tid & 127); bq[k] = j < Ck ? bep[j] : -INFINITY; }
    // only the consumer polls the mbarrier; everyone else sleeps at the hardware barrier
    if (warp == 1) {
      if (!tc::mbar_wait(&bars.done, done_ph)) ok = false;
      tc::fence_before_sync();
    }
    ok = __syncthreads_and(ok);
    done_ph ^= 1;
    cntA += TA;
    tc::fence_after_sync();
    for (int qs = 0; qs * FQ < n; ++qs) {
      // ---- B: TMEM -> sc[r][j] for the 16 queries of this step
#pragma unroll
      for (int k = 0; k < KT; ++k) {
        const int jt = tg + NTG * k;
        if (jt >= NJ) break;
        float v[FQ];
        if constexpr (FQ == 16) tc::tmem_ld16(tbase + ((uint32_t)(lq * 32) << 16) + jt * FR + qs * FQ, v);
        else tc::tmem_ld8(tbase + ((uint32_t)(lq * 32) << 16) + jt * FR + qs * FQ, v);
        const int j = jt * kFJ + (tid & 127);
        const float b = bq[k];
#pragma unroll
        for (int r = 0; r < FQ; ++r) sc[r * CkP + j] = b == -INFINITY ? -INFINITY : fmaf(v[r], dm.sigma, b);
      }
      __syncthreads();
      // ---- C: selection + softmax of the far set; P (bf16) as a K-major operand [64][Ck]
      const int r = qs * FQ + warp;                    // one query per warp
      float* s = sc + warp * CkP;
      float sum = 0.f, mx = -INFINITY;
      float v[NKMAX];                                  // (rows past the segment's end are masked below)
      const int NK = CkP >> 5;
      if (r < n) {
        const int t = rows[r];
        int32_t* so = sel_out + ((size_t)pq * dm.N + t) * m;
        if (sel_in != nullptr || dm.sel_mode == MUSE_SEL_PER_QCLUSTER) {
          const int32_t* si = sel_in != nullptr ? sel_in + ((size_t)pq * dm.N + t) * m : selq;
          for (int k = lane; k < m; k += 32) { int c = si[k]; c = (c >= 0 && c < Ck) ? c : -1; so[k] = c; if (c >= 0) s[c] = -INFINITY; }
          __syncwarp();
          load_scores<NKMAX>(s, NK, lane, v);
        } else {
          load_scores<NKMAX>(s, NK, lane, v);
          // this query's own (not yet written) P row doubles as the candidate scratch
          if (m > 0) select_top_m<NKMAX>(s, CkP, m, so, lane, Pm + r * 128, FR * 128, CkP >= 512, v);
        }
        float m4[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
        for (int k = 4; k < NKMAX; ++k) m4[k & 3] = fmaxf(m4[k & 3], v[k]);
        mx = warp_max(fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])));
      }
      __syncwarp();                                    // (the candidates have been read: P takes their place)
      // probabilities, four consecutive clusters (eight bytes) at a time
      const bool some = mx != -INFINITY;
#pragma unroll
      for (int k = 0; k < NKMAX; k += 4) {
        if (k >= NK) break;
        uint32_t w[2] = {0u, 0u};
        if (some) {
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const __nv_bfloat162 b = __floats2bfloat162_rn(__expf(v[k + 2 * e] - mx), __expf(v[k + 2 * e + 1] - mx));
            sum += __low2float(b) + __high2float(b);
            w[e] = *reinterpret_cast<const uint32_t*>(&b);
          }
        }
        const int q = (4 * lane + 32 * k) >> 3;
        *reinterpret_cast<uint2*>(Pm + (q >> 3) * (FR * 128) + tc::sw128_off(r, q & 7) + 8 * (lane & 1)) = make_uint2(w[0], w[1]);
      }
      sum = warp_sum(sum);
      if (lane == 0) {
        rinv[r] = sum > 0.f ? 1.f / sum : 0.f;
        if (r < n) lse_far[(size_t)pq * dm.N + rows[r]] = sum > 0.f ? mx + logf(sum) : -INFINITY;
      }
      __syncthreads();
    }
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    // ---- D: out^T = nu^T P^T, nu by units through the score region and the part of P that has been used
    const int NU = CkP / KU;
    if (prod >= 0 && ok) {
      for (int u = prod; u < NU; u += 4) {
        if (after_s[u] >= 0 && !tc::mbar_wait(&bars.emptyD[after_s[u]], phD)) { ok = false; break; }
        const int s = slot_s[u], n0 = sc_bytes / kSlot;
        unsigned char* dst = s < n0 ? sm + p_bytes + s * kSlot : sm + (s - n0) * kSlot;
        tc::mbar_expect_tx_warp(&bars.fullD[u], kSlot);
        for (int g = 0; g < G; ++g) tc::tma_load_3d_warp(dst + g * KU * 128, &tm_nu, 64 * g, u * KU, seg, &bars.fullD[u]);
      }
    } else if (warp == 1 && ok) {
      tc::fence_after_sync();
      // M = 128 output dims even when D = 64: the second 64-dim group of the MN-major operand then reads whatever
      // follows the unit in shared memory, and output lanes 64..127 hold numbers that nobody reads
      const uint32_t idesc = tc::idesc_bf16(128, FR, 1, 0);
      const uint64_t dp0 = tc::smem_desc_sw128(tc::smem_u32(Pm), 16, 1024);
      const uint64_t dn0 = tc::smem_desc_sw128(tc::smem_u32(sm), KU * 128, 1024);
      for (int u = 0; u < NU; ++u) {
        const int s = slot_s[u], n0 = sc_bytes / kSlot;
        const uint64_t da = tc::desc_step(dn0, (uint32_t)(s < n0 ? p_bytes + s * kSlot : (s - n0) * kSlot)), dp = tc::desc_step(dp0, (uint32_t)(u * (KU / 64)) * (FR * 128));
        if (!tc::mbar_wait(&bars.fullD[u], phD)) { ok = false; break; }
#pragma unroll
        for (int ks = 0; ks < KU / 16; ++ks)
          tc::mma_bf16_ss_warp(tbase, tc::desc_step(da, ks * 16 * 128), tc::desc_step(dp, (ks / 4) * (FR * 128) + (ks % 4) * 32), idesc,
                          u > 0 || ks > 0);
        tc::mma_commit_warp(&bars.emptyD[u]);
      }
      if (ok) tc::mma_commit_warp(&bars.done);
    }
    if (warp == 1) {
      if (!tc::mbar_wait(&bars.done, done_ph)) ok = false;
      tc::fence_before_sync();
    }
    ok = __syncthreads_and(ok);
    done_ph ^= 1;
    phD ^= 1;
    tc::fence_after_sync();
    // ---- E: thread = output dim d; warps 0-3 read queries 0..31, warps 4-7 queries 32..63
    if (warp < FR / 8) {
      const int half = warp >> 2;
      float v[32];
      tc::tmem_ld32(tbase + ((uint32_t)(lq * 32) << 16) + 32 * half, v);
      if (ok && (tid & 127) < D) {
#pragma unroll
        for (int r = 0; r < 32; ++r)
          if (32 * half + r < n) o_far[((size_t)pq * dm.N + rows[32 * half + r]) * D + (tid & 127)] = v[r] * rinv[32 * half + r];
      }
    }
    tc::fence_before_sync();
    __syncthreads();
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tbase, tcols);
  if (!ok && tid == 0) report_status(status, 3);
}

bool far_fwd_tc_supported(const Dims& d, int dtype) {
  return dtype == MUSE_BF16 && (d.D == 64 || d.D == 128) && d.Ck <= 2048;
}

bool far_fwd_small_supported(const Dims& d, bool sel_given);
int far_fwd_small(const Dims& d, const SummPtrs& sp, const void* Q, const int32_t* off_q, const int32_t* perm_q, const int32_t* sel_in,
                  int32_t* sel_out, float* o_far, float* lse_far, int* status, cudaStream_t st);

int far_fwd_tc(const Dims& d, const SummPtrs& sp, const void* Q, const int32_t* off_q, const int32_t* perm_q,
               const int32_t* sel_in, int32_t* sel_out, float* o_far, float* lse_far, int* status, cudaStream_t st) {
  // four threads per query hold their scores and a sorted list of the largest in registers up to 256 clusters and lists of 16
  if (far_fwd_small_supported(d, sel_in != nullptr)) return far_fwd_small(d, sp, Q, off_q, perm_q, sel_in, sel_out, o_far, lse_far, status, st);
  // [segments][Ck][D]
  const uint64_t dims[3] = {(uint64_t)d.D, (uint64_t)d.Ck, (uint64_t)d.B * d.Hq * d.SB * d.Cq};
  const uint64_t strides[2] = {(uint64_t)d.D * 2, (uint64_t)d.Ck * d.D * 2};
  const uint32_t box[3] = {64, kFJ, 1}, box_nu[3] = {64, (uint32_t)(kSlot / (d.D * 2)), 1};
  CUtensorMap khi, klo, nu;
  MUSE_RC(make_tmap_bf16_nd(&khi, sp.khi, 3, dims, strides, box));
  MUSE_RC(make_tmap_bf16_nd(&klo, sp.klo, 3, dims, strides, box));
  MUSE_RC(make_tmap_bf16_nd(&nu, sp.nu, 3, dims, strides, box_nu));
  const int CkP = cdiv(d.Ck, kFJ) * kFJ;
  const bool wide = d.Ck > 1024;                                         // 32 queries per pass, 8 per selection step
  const int FR = wide ? 32 : 64, FQ = wide ? 8 : 16;
  const int tile_bytes = kFJ * d.D * 2;
  const int p_bytes = FR * CkP * 2;                                    // P: bf16 [FR][Ck]
  int sc_bytes = FQ * CkP * 4;                                         // FQ score rows, later nu
  if (sc_bytes < 2 * tile_bytes) sc_bytes = 2 * tile_bytes;
  int nsA = (p_bytes + sc_bytes) / tile_bytes;
  nsA = nsA > kMaxStA ? kMaxStA : nsA;
  // (D = 64: one more tile of room behind the ring, which the padded 128-row products of phase D read past)
  const size_t smem = (size_t)p_bytes + sc_bytes + FR * d.D * 2 + 1024 + (d.D == 64 ? tile_bytes : 0);
  prof_mark("k_far_fwd_tc", st, "k_far_fwd_tc");
  // TMEM columns: all FR x Ck scores of a pass (the output of phase D reuses them), a power of two >= 32
  int tcols = 32;
  while (tcols < FR * (CkP / kFJ)) tcols *= 2;
#define MUSE_FAR_FWD_LAUNCH(FR_, FQ_, D_, NK_, MB_)                                                                              \
  do {                                                                                                                         \
    MUSE_RC(launch_pdl(k_far_fwd_tc<FR_, FQ_, D_, NK_, MB_>, dim3(d.Cq, d.SB, d.B * d.Hq), FQ_ * 32, smem, st,                     \
        d, khi, klo, nu, (const bf16*)Q, off_q, perm_q, sp.mu, sp.beta, sel_in, sel_out, o_far, lse_far, p_bytes, sc_bytes, nsA, tcols, status));   \
  } while (0)
  if (wide) { if (d.D == 128) MUSE_FAR_FWD_LAUNCH(32, 8, 128, 64, 1); else MUSE_FAR_FWD_LAUNCH(32, 8, 64, 64, 1); }
  else if (d.Ck <= 256) { if (d.D == 128) MUSE_FAR_FWD_LAUNCH(64, 16, 128, 8, 2); else MUSE_FAR_FWD_LAUNCH(64, 16, 64, 8, 2); }
  else { if (d.D == 128) MUSE_FAR_FWD_LAUNCH(64, 16, 128, 32, 1); else MUSE_FAR_FWD_LAUNCH(64, 16, 64, 32, 1); }
#undef MUSE_FAR_FWD_LAUNCH
  MUSE_LAUNCH_OK();
  return MUSE_OK;
}

}  // namespace muse
