// Far-field forward on the tensor cores for few key clusters (Ck <= 256) and short selections (m <= 16, or selections that
// are given); far_fwd_tc.cu has the definitions and the kernel for the rest.  One CTA per (query cluster i, plane, head)
// segment, 64 of its queries per pass:
//   A  scores^T[j][r] = (kappa_hi[j] + kappa_lo[j]) . q[r]   clusters on the M side (tiles of 128), queries on the N side;
//      all of the segment's kappa and nu tiles arrive by TMA at the start
//   B  tensor memory -> shared memory, transposed to [r][j] fp32, beta added
//   C  four threads per query, a quarter of its scores each in registers: a running sorted list of the largest (branch-free
//      max / min steps) per thread, two merges, and everything above the m-th largest is selected (ties: lowest cluster
//      first); softmax over the rest, P written as a bf16 operand
//   D  out^T[d][r] = sum_j nu[j][d] P[r][j]
// A warp per query, which the other kernel has, takes some thousand instructions per query for the bisection to the m-th
// largest score and its votes; four threads per query take 2 * Ck / 4 * 8 (or 16) max / min steps for eight queries at once.
//
// Bound by the latency of the phases; several CTAs share an SM.  MEASURED
#include <cuda.h>
#include "common.cuh"
#include "tc05.cuh"

namespace muse {

typedef __nv_bfloat16 bf16;
int make_tmap_bf16_nd(void* out_map, const void* base, int rank, const uint64_t* dims, const uint64_t* strides_bytes, const uint32_t* box);

namespace fs {
constexpr int kJ = 128, kR = 64, kThreads = 256;           // clusters of a tile, queries of a pass
template <int D, int CT> struct Lay {                      // CT: tiles of clusters
  static constexpr int kTile = kJ * D * 2, LD = CT * kJ + 4;                  // LD: floats per score row (16-byte reads of 8 rows do not conflict)
  static constexpr int kKappa = 2 * CT * kTile, kScore = kR * LD * 4, kArea = kKappa > kScore ? kKappa : (kScore + 1023) / 1024 * 1024;
  // at D = 64 the 128-row products of phase D read one tile past nu, into the area behind it, and ignore the result
  static constexpr int oNu = 0, oArea = CT * kTile, oQ = oArea + kArea, total = oQ + kR * D * 2 + 1024;
  static constexpr int kMin = total <= 75 * 1024 ? 3 : total <= 113 * 1024 ? 2 : 1;      // CTAs per SM
};
struct Bars { uint64_t kappa, nu, done; };
}  // namespace fs

template <int D, int CT, int ML>
__global__ void __launch_bounds__(fs::kThreads, fs::Lay<D, CT>::kMin)
k_far_fwd_small(Dims dm, const __grid_constant__ CUtensorMap tm_khi, const __grid_constant__ CUtensorMap tm_klo, const __grid_constant__ CUtensorMap tm_nu,
                const bf16* __restrict__ Q, const int32_t* __restrict__ off_q, const int32_t* __restrict__ perm_q, const float* __restrict__ mu,
                const float* __restrict__ beta, const int32_t* __restrict__ sel_in, int32_t* __restrict__ sel_out, float* __restrict__ o_far,
                float* __restrict__ lse_far, int* __restrict__ status) {
  using namespace fs;
  typedef Lay<D, CT> LY;
  constexpr int G = D / 64, kTile = LY::kTile, LD = LY::LD, NV = 32 * CT;     // NV: scores per thread
  constexpr uint32_t kCols = 64 * CT;
  extern __shared__ __align__(1024) unsigned char sm_raw[];
  __shared__ Bars bars;
  __shared__ uint32_t tbase_s;
  __shared__ int32_t rows[kR], selq[kMaxM];
  __shared__ float rinv[kR], tmp[CT * kJ];
  const int i = blockIdx.x, pl = blockIdx.y, pq = blockIdx.z, blk = dm.causal ? pl + 1 : 0, Ck = dm.Ck, m = dm.m;
  const int tid = threadIdx.x, warp = tc::warp_index(), lane = tid & 31;
  unsigned char* sm = sm_raw + ((1024u - (tc::smem_u32(sm_raw) & 1023u)) & 1023u);
  float* sc = reinterpret_cast<float*>(sm + LY::oArea);
  unsigned char *Pm = sm + LY::oArea, *Qs = sm + LY::oQ;
  if (warp == 0) tc::tmem_alloc(&tbase_s, kCols);
  if (tid == 0) { tc::mbar_init(&bars.kappa, 1); tc::mbar_init(&bars.nu, 1); tc::mbar_init(&bars.done, 1); tc::mbar_init_fence(); }
  pdl_trigger();
  pdl_wait();
  const int32_t* oq = off_q + (size_t)pq * (dm.S * dm.Cq + 1) + (size_t)blk * dm.Cq + i;
  const int p0 = oq[0], p1 = oq[1];
  const int seg = (pq * dm.SB + pl) * dm.Cq + i;
  const size_t ent0 = (size_t)seg * Ck;
  const bf16* Qp = Q + (size_t)pq * dm.N * D;
  const int32_t* pm = perm_q + (size_t)pq * dm.N;
  const bool percluster = dm.sel_mode == MUSE_SEL_PER_QCLUSTER && sel_in == nullptr && m > 0;
  if (percluster && warp == 1) {
    // one selection per segment: clusters ranked by accumulated log-mass alone
    for (int j = lane; j < Ck; j += 32) tmp[j] = mu[ent0 + j];
    __syncwarp();
    for (int k = 0; k < m; ++k) {
      float bv = -INFINITY;
      int bi = 0x7fffffff;
      for (int j = lane; j < Ck; j += 32)
        if (tmp[j] > bv) { bv = tmp[j]; bi = j; }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
      }
      if (lane == 0) selq[k] = bv == -INFINITY ? -1 : bi;
      if (bv != -INFINITY && (bi & 31) == lane) tmp[bi] = -INFINITY;
      __syncwarp();
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tbase = tbase_s;
  bool ok = true;
  uint32_t done_ph = 0, k_ph = 0;
  for (int r0 = p0; r0 < p1 && ok; r0 += kR) {
    const int n = min(kR, p1 - r0), n16 = (n + 15) & ~15;
    if (warp == 0) {                                       // ---- A
      tc::mbar_expect_tx_warp(&bars.kappa, 2 * CT * kTile);
#pragma unroll
      for (int t = 0; t < CT; ++t)
#pragma unroll
        for (int g = 0; g < G; ++g) {
          tc::tma_load_3d_warp(sm + LY::oArea + 2 * t * kTile + g * kJ * 128, &tm_khi, 64 * g, t * kJ, seg, &bars.kappa);
          tc::tma_load_3d_warp(sm + LY::oArea + (2 * t + 1) * kTile + g * kJ * 128, &tm_klo, 64 * g, t * kJ, seg, &bars.kappa);
        }
      if (r0 == p0) {
        tc::mbar_expect_tx_warp(&bars.nu, CT * kTile);
#pragma unroll
        for (int t = 0; t < CT; ++t)
#pragma unroll
          for (int g = 0; g < G; ++g) tc::tma_load_3d_warp(sm + LY::oNu + t * kTile + g * kJ * 128, &tm_nu, 64 * g, t * kJ, seg, &bars.nu);
      }
    }
    if (tid < kR) {
      int t = tid < n ? pm[r0 + tid] : -1;
      if (t >= 0 && !MUSE_IN_RANGE(t, dm.N)) t = -1;
      rows[tid] = t;
    }
    // query rows -> K-major swizzled tile [64][D] bf16 (G blocks of [64][128 B])
    for (int e = tid; e < n16 * (D / 8); e += kThreads) {
      const int r = e / (D / 8), ck = e % (D / 8);
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      if (r < n && MUSE_IN_RANGE(pm[r0 + r], dm.N)) v = reinterpret_cast<const uint4*>(Qp + (size_t)pm[r0 + r] * D)[ck];
      *reinterpret_cast<uint4*>(Qs + (ck >> 3) * kR * 128 + tc::sw128_off(r, ck & 7)) = v;
    }
    float bq[CT];                                          // beta of this thread's clusters (lane = cluster in phase B)
#pragma unroll
    for (int t = 0; t < CT; ++t) { const int j = t * kJ + (tid & 127); bq[t] = j < Ck ? beta[ent0 + j] : -INFINITY; }
    tc::fence_async_smem();
    __syncthreads();
    if (warp == 1) {
      if (!tc::mbar_wait(&bars.kappa, k_ph)) ok = false;
      tc::fence_after_sync();
      const uint32_t idesc = tc::idesc_bf16(kJ, n16, 0, 0);
      const uint64_t dq = tc::smem_desc_sw128(tc::smem_u32(Qs), 16, 1024), da = tc::smem_desc_sw128(tc::smem_u32(sm + LY::oArea), 16, 1024);
#pragma unroll
      for (int t = 0; t < 2 * CT; ++t)
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks)
          tc::mma_bf16_ss_warp(tbase + (t >> 1) * kR, tc::desc_step(da, t * kTile + (ks / 4) * kJ * 128 + (ks % 4) * 32),
                               tc::desc_step(dq, (ks / 4) * kR * 128 + (ks % 4) * 32), idesc, (t & 1) || ks > 0);
      tc::mma_commit_warp(&bars.done);
      if (!tc::mbar_wait(&bars.done, done_ph)) ok = false;
      tc::fence_before_sync();
    }
    k_ph ^= 1;
    ok = __syncthreads_and(ok);
    done_ph ^= 1;
    tc::fence_after_sync();
    // ---- B: the kappa tiles have been read, the scores take their place.  Warps 0-3: queries 0-31, warps 4-7: the others
#pragma unroll
    for (int t = 0; t < CT; ++t)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c0 = 32 * (warp >> 2) + 16 * h;
        if (c0 < n16) {
          float v[16];
          tc::tmem_ld16(tbase + ((uint32_t)((warp & 3) * 32) << 16) + t * kR + c0, v);
#pragma unroll
          for (int r = 0; r < 16; ++r) sc[(c0 + r) * LD + t * kJ + (tid & 127)] = bq[t] == -INFINITY ? -INFINITY : fmaf(v[r], dm.sigma, bq[t]);
        }
      }
    tc::fence_before_sync();
    __syncthreads();
    // ---- C: thread q of a query's four has its chunks q, q + 4, ... of eight clusters
    const int r = warp * 8 + (lane >> 2), q = lane & 3;
    const bool live = r < n && rows[r] >= 0;
    int32_t* so = sel_out + ((size_t)pq * dm.N + max(r < n ? rows[r] : 0, 0)) * m;
    float* s = sc + r * LD;
    if (warp * 8 < n && (sel_in != nullptr || percluster)) {
      if (live)
        for (int k = q; k < m; k += 4) {
          int c = percluster ? selq[k] : sel_in[((size_t)pq * dm.N + rows[r]) * m + k];
          c = c >= 0 && c < Ck ? c : -1;
          so[k] = c;
          if (c >= 0) s[c] = -INFINITY;
        }
      __syncwarp();
    }
    float v[NV];
    if (warp * 8 < n) {
#pragma unroll
      for (int t = 0; t < NV / 8; ++t) {
        const float4 a = *reinterpret_cast<const float4*>(s + 8 * (q + 4 * t)), b = *reinterpret_cast<const float4*>(s + 8 * (q + 4 * t) + 4);
        v[8 * t] = a.x; v[8 * t + 1] = a.y; v[8 * t + 2] = a.z; v[8 * t + 3] = a.w;
        v[8 * t + 4] = b.x; v[8 * t + 5] = b.y; v[8 * t + 6] = b.z; v[8 * t + 7] = b.w;
      }
      if (sel_in == nullptr && !percluster && m > 0) {     // (the same in every thread)
        float a[ML];                                       // the largest so far, descending
#pragma unroll
        for (int k = 0; k < ML; ++k) a[k] = -INFINITY;
#pragma unroll
        for (int e = 0; e < NV; ++e) {
          float x = v[e];
#pragma unroll
          for (int k = 0; k < ML; ++k) { const float hi = fmaxf(a[k], x); x = fminf(a[k], x); a[k] = hi; }
        }
#pragma unroll
        for (int o = 1; o <= 2; o <<= 1) {                 // merge with the neighbour's list: the larger halves form a bitonic sequence
          float b[ML];
#pragma unroll
          for (int k = 0; k < ML; ++k) b[k] = __shfl_xor_sync(0xffffffffu, a[k], o);
#pragma unroll
          for (int k = 0; k < ML; ++k) a[k] = fmaxf(a[k], b[ML - 1 - k]);
#pragma unroll
          for (int d = ML / 2; d > 0; d >>= 1)
#pragma unroll
            for (int k = 0; k < ML; ++k)
              if ((k & d) == 0) { const float hi = fmaxf(a[k], a[k + d]), lo = fminf(a[k], a[k + d]); a[k] = hi; a[k + d] = lo; }
        }
        float T = a[0];
#pragma unroll
        for (int k = 1; k < ML; ++k) T = k == m - 1 ? a[k] : T;
        uint32_t gt[CT], eq[CT];                           // above the m-th largest; equal to it (none if fewer than m are finite)
        int cnt = 0;                                       // both counts, 16 bits each
#pragma unroll
        for (int w = 0; w < CT; ++w) {
          gt[w] = eq[w] = 0u;
#pragma unroll
          for (int e = 0; e < 32; ++e) {
            gt[w] |= v[32 * w + e] > T ? 1u << e : 0u;
            eq[w] |= v[32 * w + e] == T ? 1u << e : 0u;
          }
          if (T == -INFINITY) eq[w] = 0u;
          cnt += __popc(gt[w]) | __popc(eq[w]) << 16;
        }
        int all = cnt + __shfl_xor_sync(0xffffffffu, cnt, 1);
        all += __shfl_xor_sync(0xffffffffu, all, 2);
        int need = m - (all & 0xffff);                     // ties still to take
        bool few = (all >> 16) <= need;
        if (few) {
#pragma unroll
          for (int w = 0; w < CT; ++w) gt[w] |= eq[w];
        }
        while (__any_sync(0xffffffffu, !few && need > 0)) {            // more ties than places: lowest cluster first
          int jm = 0x7fffffff;                             // (bit e of word w is cluster 8 (q + 4 (4 w + e / 8)) + e % 8: ascending)
#pragma unroll
          for (int w = CT - 1; w >= 0; --w)
            if ((eq[w] & ~gt[w]) != 0u) { const int e = __ffs((int)(eq[w] & ~gt[w])) - 1; jm = 8 * (q + 4 * (4 * w + (e >> 3))) + (e & 7); }
          int jq = min(jm, __shfl_xor_sync(0xffffffffu, jm, 1));
          jq = min(jq, __shfl_xor_sync(0xffffffffu, jq, 2));
          if (!few && need > 0 && jm == jq) {
            const int ch = jm >> 5, e = (ch & 3) * 8 + (jm & 7);       // chunk (jm >> 3) = q + 4 ch
#pragma unroll
            for (int w = 0; w < CT; ++w) if ((ch >> 2) == w) gt[w] |= 1u << e;
          }
          --need;
        }
        int mine = 0;
#pragma unroll
        for (int w = 0; w < CT; ++w) mine += __popc(gt[w]);
        int inc = mine;
        { const int x = __shfl_up_sync(0xffffffffu, inc, 1, 4); if (q >= 1) inc += x; }
        { const int x = __shfl_up_sync(0xffffffffu, inc, 2, 4); if (q >= 2) inc += x; }
        const int tot = __shfl_sync(0xffffffffu, inc, 3, 4);
        if (live) {
          int at = inc - mine;
#pragma unroll
          for (int w = 0; w < CT; ++w)
            for (uint32_t b = gt[w]; b != 0u; b &= b - 1u) {
              const int e = __ffs((int)b) - 1;
              if (at < m) so[at] = 8 * (q + 4 * (4 * w + (e >> 3))) + (e & 7);
              ++at;
            }
          for (int k = tot + q; k < m; k += 4) so[k] = -1;
        }
#pragma unroll
        for (int e = 0; e < NV; ++e) v[e] = (gt[e >> 5] >> (e & 31)) & 1u ? -INFINITY : v[e];
      }
    }
    __syncthreads();                                       // every score has been read: P takes their place
    if (warp * 8 < n16) {
      float mx = -INFINITY, sum = 0.f;
      if (live) {
#pragma unroll
        for (int e = 0; e < NV; ++e) mx = fmaxf(mx, v[e]);
      }
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
#pragma unroll
      for (int t = 0; t < NV / 8; ++t) {
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          float a = 0.f, b = 0.f;
          if (mx != -INFINITY) { a = __expf(v[8 * t + 2 * k] - mx); b = __expf(v[8 * t + 2 * k + 1] - mx); }
          const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
          sum += __low2float(h) + __high2float(h);
          w[k] = *reinterpret_cast<const uint32_t*>(&h);
        }
        const int ch = q + 4 * t;
        *reinterpret_cast<uint4*>(Pm + (ch >> 3) * (kR * 128) + tc::sw128_off(r, ch & 7)) = make_uint4(w[0], w[1], w[2], w[3]);
      }
      sum += __shfl_xor_sync(0xffffffffu, sum, 1);
      sum += __shfl_xor_sync(0xffffffffu, sum, 2);
      if (q == 0) {
        rinv[r] = sum > 0.f ? 1.f / sum : 0.f;
        if (live) lse_far[(size_t)pq * dm.N + rows[r]] = sum > 0.f ? mx + logf(sum) : -INFINITY;
      }
    }
    tc::fence_async_smem();
    __syncthreads();
    // ---- D (all threads' reads of the scores in tensor memory are behind them)
    if (warp == 1) {
      if (r0 == p0 && !tc::mbar_wait(&bars.nu, 0)) ok = false;
      tc::fence_after_sync();
      const uint32_t idesc = tc::idesc_bf16(128, n16, 1, 0);
      const uint64_t dp = tc::smem_desc_sw128(tc::smem_u32(Pm), 16, 1024), dn = tc::smem_desc_sw128(tc::smem_u32(sm + LY::oNu), kJ * 128, 1024);
#pragma unroll
      for (int t = 0; t < CT; ++t)
#pragma unroll
        for (int ks = 0; ks < kJ / 16; ++ks)
          tc::mma_bf16_ss_warp(tbase, tc::desc_step(dn, t * kTile + ks * 16 * 128), tc::desc_step(dp, 2 * t * (kR * 128) + (ks / 4) * (kR * 128) + (ks % 4) * 32),
                               idesc, t > 0 || ks > 0);
      tc::mma_commit_warp(&bars.done);
      if (!tc::mbar_wait(&bars.done, done_ph)) ok = false;
      tc::fence_before_sync();
    }
    ok = __syncthreads_and(ok);
    done_ph ^= 1;
    tc::fence_after_sync();
    // ---- E: thread = output dim; warps 0-3 queries 0-31, warps 4-7 the others
    if (32 * (warp >> 2) < n && (warp & 3) * 32 < D) {
      const int h = 32 * (warp >> 2);
      float x[32];
      tc::tmem_ld32(tbase + ((uint32_t)((warp & 3) * 32) << 16) + h, x);
      if (ok) {
#pragma unroll
        for (int k = 0; k < 32; ++k)
          if (h + k < n && rows[h + k] >= 0) o_far[((size_t)pq * dm.N + rows[h + k]) * D + (tid & 127)] = x[k] * rinv[h + k];
      }
    }
    tc::fence_before_sync();
    __syncthreads();
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tbase, kCols);
  if (!ok && tid == 0) report_status(status, 3);
}

bool far_fwd_small_supported(const Dims& d, bool sel_given) {
  return d.Ck <= 256 && (d.m <= 16 || sel_given || d.sel_mode == MUSE_SEL_PER_QCLUSTER);
}

template <int D, int CT, int ML>
static int far_fwd_small_t(const Dims& d, const CUtensorMap& khi, const CUtensorMap& klo, const CUtensorMap& nu, const SummPtrs& sp, const void* Q,
                           const int32_t* off_q, const int32_t* perm_q, const int32_t* sel_in, int32_t* sel_out, float* o_far, float* lse_far,
                           int* status, cudaStream_t st) {
  return launch_pdl(k_far_fwd_small<D, CT, ML>, dim3(d.Cq, d.SB, d.B * d.Hq), fs::kThreads, fs::Lay<D, CT>::total, st, d, khi, klo, nu, (const bf16*)Q,
                    off_q, perm_q, sp.mu, sp.beta, sel_in, sel_out, o_far, lse_far, status);
}

int far_fwd_small(const Dims& d, const SummPtrs& sp, const void* Q, const int32_t* off_q, const int32_t* perm_q, const int32_t* sel_in,
                  int32_t* sel_out, float* o_far, float* lse_far, int* status, cudaStream_t st) {
  // [segments][Ck][D]; rows of the last tile past Ck are zeros
  const uint64_t dims[3] = {(uint64_t)d.D, (uint64_t)d.Ck, (uint64_t)d.B * d.Hq * d.SB * d.Cq};
  const uint64_t strides[2] = {(uint64_t)d.D * 2, (uint64_t)d.Ck * d.D * 2};
  const uint32_t box[3] = {64, fs::kJ, 1};
  CUtensorMap khi, klo, nu;
  MUSE_RC(make_tmap_bf16_nd(&khi, sp.khi, 3, dims, strides, box));
  MUSE_RC(make_tmap_bf16_nd(&klo, sp.klo, 3, dims, strides, box));
  MUSE_RC(make_tmap_bf16_nd(&nu, sp.nu, 3, dims, strides, box));
  prof_mark("k_far_fwd_tc", st);
  const bool two = d.Ck > fs::kJ, long_list = d.m > 8;
#define MUSE_FS(D_, CT_, ML_) far_fwd_small_t<D_, CT_, ML_>(d, khi, klo, nu, sp, Q, off_q, perm_q, sel_in, sel_out, o_far, lse_far, status, st)
  if (d.D == 128) return two ? (long_list ? MUSE_FS(128, 2, 16) : MUSE_FS(128, 2, 8)) : (long_list ? MUSE_FS(128, 1, 16) : MUSE_FS(128, 1, 8));
  return two ? (long_list ? MUSE_FS(64, 2, 16) : MUSE_FS(64, 2, 8)) : (long_list ? MUSE_FS(64, 1, 16) : MUSE_FS(64, 1, 8));
#undef MUSE_FS
}

}  // namespace muse
