// Exact causal attention inside the spatial blocks, forward (Section "Exact Retrieval and Local Attention"), bf16
// inputs, D = 64 or 128.  A CTA owns two consecutive tiles of 128 queries of one block and walks the block's keys up to
// them in tiles of 128:
//   S_q = Q_q K^T        tcgen05.mma, both operands K-major in shared memory (TMA), accumulator in tensor memory
//   P_q                  two threads per query row, 64 keys each: exponentials, bf16; written over the consumed logits
//                        in tensor memory, from where it is the A operand of
//   O_q += P_q V         accumulated in tensor memory over all key tiles, rescaled lazily
// The (query tile, key tile) pairs, numbered n = 2 t + q, go through NB logit buffers in turn.  While the eight warps of
// one query tile are at their exponentials the tensor cores work on the other, and with NB = 3 (D = 64, where the outputs
// leave room) a query tile's next logits are there when its warps come back for them.  One warp issues every product,
// one every load.
//
// Products are issued in the order ... O += P(n) V, S(n + NB) = Q K ..., and the tensor core executes a CTA's products in
// the order they were issued, so S(n + NB) may overwrite P(n).
//
// Bound by the exponentials at D = 64 (16 per clock and SM: 2048 cycles per pair of 128 x 128 tiles against 1300 of MMA),
// by both alike at D = 128 (2048 and 2048), and in practice by the latency of one warp's pass over its logits (a warp or two
// per scheduler): two threads per row and NB = 3 took D = 64 from 3990 (one thread, NB = 2) to 3300 us at 32 heads of 64k
// tokens, at D = 128 two threads per row were slower (638 -> 1060 us) and there is no room for a third buffer.
// Against one 128-query tile per CTA with P through shared memory and a CTA barrier per tile: 64k tokens in 8 blocks,
// D = 64, 32 heads 5926 -> 3300 us (667 TFLOP/s); D = 128, 4 heads 908 -> 638 us (862); 128k tokens, 4 heads 3400 ->
// 2290 us (960).  Since then two logits per instruction where one rounds like the other, three per maximum and no spills around the
// rescaling: 32 heads, D = 64 3600 -> 3000 us; 4 heads, D = 128 637 -> 505.
#include <cuda.h>
#include "common.cuh"
#include "tc05.cuh"

namespace muse {

typedef __nv_bfloat16 bf16;
int make_tmap_bf16_rows(void* out_map, const void* base, uint64_t rows, uint32_t cols, uint32_t box_rows);

namespace lf {
constexpr int kRows = 128, kKeys = 128;
template <int D> struct Lay {
  static constexpr int kTile = 128 * D * 2, kStages = D == 128 ? 2 : 3, NB = D == 128 ? 2 : 3;
  static constexpr int H = D == 128 ? 1 : 2, kSoft = 256 * H, kThreads = kSoft + 64;    // threads per query row; softmax threads, an MMA warp, a load warp
  static constexpr int oQ = 0, oK = 2 * kTile, oV = oK + kStages * kTile, total = oV + kStages * kTile + 1024;
};
struct Bars { uint64_t q_full[2], k_full[3], k_empty[3], v_full[3], v_empty[3], s_full[3], p_ready[2], pv_done[2]; };

// barrier among `count` threads with an OR of their predicates
__device__ __forceinline__ bool bar_or(int id, int count, bool p) {
  uint32_t r;
  asm volatile("{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbarrier.cta.red.or.pred q, %2, %3, p;\nselp.u32 %0, 1, 0, q;\n}\n"
               : "=r"(r) : "r"((uint32_t)p), "r"(id), "r"(count) : "memory");
  return r != 0;
}
}  // namespace lf

template <int D>
__global__ void __launch_bounds__(lf::Lay<D>::kThreads, 1)
k_local_fwd_tc(Dims dm, const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
               float* __restrict__ o_loc, float* __restrict__ lse_loc, int* __restrict__ status) {
  using namespace lf;
  typedef Lay<D> LY;
  constexpr int kTile = LY::kTile, NS = LY::kStages, NB = LY::NB, H = LY::H, kSoft = LY::kSoft, MW = kSoft / 32, G = D / 64;     // MW: the MMA warp
  constexpr uint32_t cO = NB * kKeys;                      // tensor-memory columns: NB logit buffers | O_0 | O_1
  extern __shared__ __align__(1024) unsigned char sm_raw[];
  __shared__ Bars bars;
  __shared__ uint32_t tbase_s;
  __shared__ float mx_s[2][2][kRows];
  const int tid = threadIdx.x, warp = tc::warp_index();
  unsigned char* sm = sm_raw + ((1024u - (tc::smem_u32(sm_raw) & 1023u)) & 1023u);
  if (warp == MW) tc::tmem_alloc(&tbase_s, 512);
  if (tid == 0) {
    for (int q = 0; q < 2; ++q) {
      tc::mbar_init(&bars.q_full[q], 1); tc::mbar_init(&bars.p_ready[q], kSoft / 2); tc::mbar_init(&bars.pv_done[q], 1);
    }
    for (int b = 0; b < NB; ++b) tc::mbar_init(&bars.s_full[b], 1);
    for (int s = 0; s < NS; ++s) {
      tc::mbar_init(&bars.k_full[s], 1); tc::mbar_init(&bars.k_empty[s], 1); tc::mbar_init(&bars.v_full[s], 1); tc::mbar_init(&bars.v_empty[s], 1);
    }
    tc::mbar_init_fence();
  }
  const int tpb = cdiv(dm.Bs, 2 * kRows);
  // heaviest tiles (latest in a block) first
  const int lin = blockIdx.x, qt = tpb - 1 - lin / dm.S, blk = lin % dm.S, pq = blockIdx.y;
  const int b_ = pq / dm.Hq, h = pq % dm.Hq, pk = b_ * dm.Hkv + dm.hm.g[h];
  const int bstart = blk * dm.Bs, bend = bstart + dm.Bs, q0 = bstart + qt * 2 * kRows;
  // key tiles of each query tile (causal: up to its last row)
  const int nq0 = min(kRows, bend - q0), nq1 = max(0, min(kRows, bend - q0 - kRows));
  const int T0 = (q0 + nq0 - bstart + kKeys - 1) / kKeys, T1 = nq1 > 0 ? (q0 + kRows + nq1 - bstart + kKeys - 1) / kKeys : 0;
  const int T = max(T0, T1);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tbase = tbase_s;
  bool ok = true;
  pdl_wait();
  pdl_trigger();

  if (warp == MW + 1) {                                         // ---- loads
    auto load = [&](unsigned char* dst, const void* map, int row, uint64_t* bar) {
      if (tc::elect_one()) {
        tc::mbar_expect_tx(bar, kTile);
#pragma unroll
        for (int g = 0; g < G; ++g) tc::tma_load_2d(dst + g * 128 * 128, map, 64 * g, row, bar);
      }
    };
    load(sm + LY::oQ, &tm_q, pq * dm.N + q0, &bars.q_full[0]);
    if (T1 > 0) load(sm + LY::oQ + kTile, &tm_q, pq * dm.N + q0 + kRows, &bars.q_full[1]);
    // (rows past the block's visible keys are loaded too; they are masked)
    for (int t = 0, s = 0, ph = 0; t < T && ok; ++t) {
      const int row = pk * dm.N + bstart + t * kKeys;
      if (!tc::mbar_wait(&bars.k_empty[s], ph ^ 1)) { ok = false; break; }
      load(sm + LY::oK + s * kTile, &tm_k, row, &bars.k_full[s]);
      if (!tc::mbar_wait(&bars.v_empty[s], ph ^ 1)) { ok = false; break; }
      load(sm + LY::oV + s * kTile, &tm_v, row, &bars.v_full[s]);
      if (++s == NS) { s = 0; ph ^= 1; }
    }
  } else if (warp == MW) {                                  // ---- products
    const uint32_t id_s = tc::idesc_bf16(kRows, kKeys, 0, 0), id_o = tc::idesc_bf16(kRows, D, 0, 1);
    const uint64_t dq = tc::smem_desc_sw128(tc::smem_u32(sm + LY::oQ), 16, 1024), dk = tc::smem_desc_sw128(tc::smem_u32(sm + LY::oK), 16, 1024),
                   dv = tc::smem_desc_sw128(tc::smem_u32(sm + LY::oV), kKeys * 128, 1024);
    int sk = 0, phk = 0;                                   // ring position of the next key tile
    bool k_in = false;                                     // ... already waited for (the first query tile has used it)
    auto issue_s = [&](int n) {                            // S(n) into buffer n % NB, where the pair exists
      const int q = n & 1, t = n >> 1;
      if (t >= T) return;
      if (!k_in) {
        if (!tc::mbar_wait(&bars.k_full[sk], phk)) { ok = false; return; }
        tc::fence_after_sync();
        k_in = true;
      }
      if (t < (q == 0 ? T0 : T1)) {
        const uint32_t cs = tbase + (uint32_t)(n % NB) * kKeys;
        const uint64_t a = tc::desc_step(dq, q * kTile), b = tc::desc_step(dk, (uint32_t)sk * kTile);
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks)
          tc::mma_bf16_ss_warp(cs, tc::desc_step(a, (ks / 4) * 128 * 128 + (ks % 4) * 32), tc::desc_step(b, (ks / 4) * 128 * 128 + (ks % 4) * 32),
                               id_s, ks > 0);
      }
      tc::mma_commit_warp(&bars.s_full[n % NB]);           // (also for a pair that does not exist: a buffer's uses stay NB pairs apart)
      if (q == 1) { tc::mma_commit_warp(&bars.k_empty[sk]); k_in = false; if (++sk == NS) { sk = 0; phk ^= 1; } }
    };
    if (!tc::mbar_wait(&bars.q_full[0], 0)) ok = false;
    if (T1 > 0 && !tc::mbar_wait(&bars.q_full[1], 0)) ok = false;
    tc::fence_after_sync();
    for (int n = 0; n < NB && ok; ++n) issue_s(n);
    for (int n = 0, s = 0, ph = 0; n < 2 * T && ok; ++n) {
      const int q = n & 1, t = n >> 1;
      if (t < (q == 0 ? T0 : T1)) {
        if (!tc::mbar_wait(&bars.p_ready[q], t & 1)) { ok = false; break; }
        if (!tc::mbar_wait(&bars.v_full[s], ph)) { ok = false; break; }
        tc::fence_after_sync();
        const uint64_t b = tc::desc_step(dv, (uint32_t)s * kTile);
        const uint32_t cp = tbase + (uint32_t)(n % NB) * kKeys;
#pragma unroll
        for (int ks = 0; ks < kKeys / 16; ++ks)
          tc::mma_bf16_ts_warp(tbase + cO + q * D, cp + 8 * ks, tc::desc_step(b, ks * 16 * 128), id_o, t > 0 || ks > 0);
        tc::mma_commit_warp(&bars.pv_done[q]);
      }
      issue_s(n + NB);
      if (q == 1) { tc::mma_commit_warp(&bars.v_empty[s]); if (++s == NS) { s = 0; ph ^= 1; } }
    }
  } else {                                                 // ---- softmax: thread = query row, or (query row, half of the tile's keys)
    constexpr int W = kKeys / H, OD = D / H;               // logits and output dims of a thread
    const int q = warp / (4 * H), half = H == 2 ? (warp >> 2) & 1 : 0, row = tid & 127, Tq = q == 0 ? T0 : T1;
    const int qrow = q0 + q * kRows + row;
    const uint32_t tl = tbase + ((uint32_t)((warp & 3) * 32) << 16), to = tl + cO + q * D + half * OD;
    const float scale2 = dm.sigma * 1.4426950408889634f;
    const uint64_t sc2 = tc::pair(scale2, scale2);
    // m2 is the exponent base in use for this row (log2 units): it follows the running maximum lazily, only when that has
    // grown by more than kLazy (probabilities then stay below 2^kLazy), and only then is the accumulator rescaled.
    constexpr float kLazy = 8.f;
    float m2 = -INFINITY, l = 0.f;                         // l: this half's share of the row sum
    for (int t = 0, b = q, bph = 0; t < Tq; ++t) {
      if (!tc::mbar_wait(&bars.s_full[b], bph)) ok = false;
      tc::fence_after_sync();
      const uint32_t ts = tl + b * kKeys;
      b += 2;
      if (b >= NB) { b -= NB; bph ^= 1; }
      float s[W / 16][16];
#pragma unroll
      for (int g = 0; g < W / 16; ++g) tc::tmem_ld16_issue(ts + W * half + 16 * g, s[g]);
      tc::tmem_ld_wait();
#pragma unroll
      for (int g = 0; g < W / 16; ++g) tc::tmem_ld_use16(s[g]);
      if (t == Tq - 1) {                                   // (earlier tiles are visible to every row)
        const int lim = qrow - (bstart + t * kKeys) - W * half;
#pragma unroll
        for (int g = 0; g < W / 16; ++g)
#pragma unroll
          for (int i = 0; i < 16; ++i) s[g][i] = 16 * g + i <= lim ? s[g][i] : -INFINITY;
      }
      float mx[W / 16];                                    // (three at a time)
#pragma unroll
      for (int g = 0; g < W / 16; ++g) {
        mx[g] = fmaxf(s[g][0], s[g][1]);
#pragma unroll
        for (int i = 2; i < 16; i += 2) mx[g] = tc::max3(mx[g], s[g][i], s[g][i + 1]);
      }
#pragma unroll
      for (int g = W / 16 - 1; g > 0; --g) mx[g - 1] = fmaxf(mx[g - 1], mx[g]);
      const float mt = mx[0] * scale2;
      // (also: both halves have read their logits before either writes P over them)
      const bool grow = t == 0 || mt > m2 + kLazy;
      if (H == 2 ? bar_or(1 + q, kSoft / 2, grow) : __any_sync(0xffffffffu, grow)) {
        float mr = mt;
        if (H == 2) {
          mx_s[q][half][row] = mt;
          tc::named_bar_sync(1 + q, kSoft / 2);
          mr = fmaxf(mt, mx_s[q][half ^ 1][row]);
        }
        const float mn = mr > m2 + kLazy ? mr : m2;                // (finite: every row sees the block's first key) rows that did not grow keep their base (factor 1)
        if (t > 0) {
          if (ok && !tc::mbar_wait(&bars.pv_done[q], (t - 1) & 1)) ok = false;
          tc::fence_after_sync();
          const float resc = tc::fast_exp2(m2 - mn);
#pragma unroll 1
          for (int d0 = 0; d0 < OD; d0 += 16) {            // (16 at a time: the logits stay in registers meanwhile)
            float v[16];
            uint32_t x[16];
            tc::tmem_ld16(to + d0, v);
#pragma unroll
            for (int i = 0; i < 16; ++i) x[i] = __float_as_uint(v[i] * resc);
            tc::tmem_st16_issue(to + d0, x);
          }
          tc::tmem_st_wait();
          l *= resc;
        }
        m2 = mn;
      }
      const float base = m2 == -INFINITY ? 0.f : m2;
      const uint64_t nb = tc::pair(-base, -base);
      uint64_t rs[4] = {0u, 0u, 0u, 0u};                   // (pairs of zeros)
#pragma unroll
      for (int g = 0; g < W / 16; ++g) {
        uint32_t pk[8];
#pragma unroll
        for (int i = 0; i < 16; i += 2) {
          float x0, x1;
          tc::unpair(tc::fma2(tc::pair(s[g][i], s[g][i + 1]), sc2, nb), x0, x1);
          const __nv_bfloat162 e2 = __floats2bfloat162_rn(tc::fast_exp2(x0), tc::fast_exp2(x1));
          pk[i / 2] = *reinterpret_cast<const uint32_t*>(&e2);
          rs[(i / 2) & 3] = tc::add2(rs[(i / 2) & 3], tc::pair_of_bf16(pk[i / 2]));      // the rounded values, as the P V product sees them
        }
        tc::tmem_st8_issue(ts + W / 2 * half + 8 * g, pk);
      }
      float l0, l1;
      tc::unpair(tc::add2(tc::add2(rs[0], rs[1]), tc::add2(rs[2], rs[3])), l0, l1);
      l += l0 + l1;
      // every phase of pv_done is waited for before the next one can complete (a wait for a phase two behind never returns)
      if (t > 0 && ok && !tc::mbar_wait(&bars.pv_done[q], (t - 1) & 1)) ok = false;
      tc::tmem_st_wait();
      tc::fence_before_sync();
      tc::mbar_arrive(&bars.p_ready[q]);
    }
    if (Tq > 0) {
      if (ok && !tc::mbar_wait(&bars.pv_done[q], (Tq - 1) & 1)) ok = false;
      tc::fence_after_sync();
      if (H == 2) {
        tc::named_bar_sync(1 + q, kSoft / 2);              // (mx_s was last read before the last tile's barrier)
        mx_s[q][half][row] = l;
        tc::named_bar_sync(1 + q, kSoft / 2);
        l += mx_s[q][half ^ 1][row];
      }
      const bool live = ok && row < (q == 0 ? nq0 : nq1);
      const size_t at = (size_t)pq * dm.N + qrow;
      const float inv = 1.f / l;
#pragma unroll
      for (int d0 = 0; d0 < OD; d0 += 32) {
        float v[32];
        tc::tmem_ld32(to + d0, v);
        if (live) {
#pragma unroll
          for (int c = 0; c < 4; ++c) {                    // 8 floats = one 32-byte sector per store
            uint32_t w[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) w[e] = __float_as_uint(v[8 * c + e] * inv);
            tc::st_global_32B(o_loc + at * D + half * OD + d0 + 8 * c, w);
          }
        }
      }
      if (live && half == 0) lse_loc[at] = (m2 + log2f(l)) * 0.6931471805599453f;
    }
  }
  if (!ok && (tid & 31) == 0) report_status(status, MUSE_STATUS_FWD_TIMEOUT);
  tc::fence_before_sync();
  __syncthreads();
  if (warp == MW) tc::tmem_dealloc(tbase, 512);
}

int local_fwd_tc(const Dims& d, const void* Q, const void* K, const void* V, float* o_loc, float* lse_loc, int* status,
                 cudaStream_t st) {
  CUtensorMap tq, tk, tv;
  MUSE_RC(make_tmap_bf16_rows(&tq, Q, (uint64_t)d.B * d.Hq * d.N, (uint32_t)d.D, lf::kRows));
  MUSE_RC(make_tmap_bf16_rows(&tk, K, (uint64_t)d.B * d.Hkv * d.N, (uint32_t)d.D, lf::kKeys));
  MUSE_RC(make_tmap_bf16_rows(&tv, V, (uint64_t)d.B * d.Hkv * d.N, (uint32_t)d.D, lf::kKeys));
  const dim3 grid(d.S * cdiv(d.Bs, 2 * lf::kRows), d.B * d.Hq);
  prof_mark("k_local_fwd_tc", st);
  if (d.D == 128) return launch_pdl(k_local_fwd_tc<128>, grid, lf::Lay<128>::kThreads, lf::Lay<128>::total, st, d, tq, tk, tv, o_loc, lse_loc, status);
  return launch_pdl(k_local_fwd_tc<64>, grid, lf::Lay<64>::kThreads, lf::Lay<64>::total, st, d, tq, tk, tv, o_loc, lse_loc, status);
}

}  // namespace muse
