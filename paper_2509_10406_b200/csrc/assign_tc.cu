// k-means assignment on the tensor cores (bf16 inputs): argmin_c |c|^2 - 2 x.c with the dot
// products from tcgen05 MMAs.  The centres are fp32; they enter the MMA as a bf16 hi + lo pair
// (two accumulating products), which keeps ~16 mantissa bits so that the discrete assignment
// agrees with an fp64 evaluation except at genuine near-ties (Appendix "Balanced Assignment":
// the |x|^2 term cancels between centres).
//
// Persistent: one CTA per SM walks a contiguous share of the work (both sides, all problems), so that barriers, tensor
// memory and the pipeline are set up once and the next points are loading while the current ones are compared.
// A unit is R = 2 tiles of 128 points of one problem: each centre tile serves both from one load.  The centre planes
// arrive as pieces of 128 centres x 64 dims (16 KB) through a ring; when all pieces of a problem fit the ring
// (C <= 512 at D = 64, C <= 128 at D = 128) they are loaded once per problem instead of once per unit.
// Small problems take R = 1, so that there are twice the units for the SMs to share.
//
// Bounds: a unit and centre tile is 32 D cycles of MMA (4096 at D = 128 with hi and lo); the arg-min costs three ALU
// instructions per distance, 1536 cycles per SM sub-partition for the two 128 x 128 tiles.  With few centres (one tile,
// D = 64) the read of the points (1400 cycles at full HBM rate) is as long as the comparison.  Measured (both sides):
// 4 heads x 65536 points, D = 128, 256 + 1024 centres 204 -> 130 us (0.80 of the MMA rate); 32 heads x 65536 points,
// D = 64, 128 + 128 centres 712 -> 144 us (3.7 TB/s).  What it took was the issuing warp: with one thread of a
// divergent branch issuing, an MMA cost about 280 cycles of that thread and the same kernel took 271 and 324 us.
#include <cuda.h>
#include "common.cuh"
#include "tc05.cuh"

namespace muse {

typedef __nv_bfloat16 bf16;
int make_tmap_bf16_rows(void* out_map, const void* base, uint64_t rows, uint32_t cols, uint32_t box_rows);

namespace at {

// Warp roles: warps 0-3 and 4-7 read the distance rows of the unit's first and second point tile, warps 8-9 load points
// and warps 10-13 centre pieces (a thread that issues a box and then waits gets 18 B/clk, four of them 70), warp 14
// issues the MMAs into two alternating accumulators per point tile.
constexpr int kXProd = 2, kCProd = 4;
constexpr int kRows = 128, kCols = kAsgTile, kThreads = (8 + kXProd + kCProd + 1) * 32, kXStages = 4, kPiece = kCols * 128, kMaxPieces = 9;

struct Bars { uint64_t xfull[kXStages], xempty[kXStages], full[kMaxPieces], empty[kMaxPieces], tfull[2][2], tempty[2][2]; };

struct Side { const float* cnorm; int32_t* assign; float* dist; const int32_t* flags; int problems, C, NT, upp; };   // upp = units per problem
struct Args { Side s[2]; int N, ns; };

// Walks the units whose cost interval starts inside this CTA's share of the total cost (a unit costs NT).
struct Walk {
  int side, prob, u; long long left;
  __device__ __forceinline__ Walk(const Args& g) {
    const long long c0 = (long long)g.s[0].problems * g.s[0].upp * g.s[0].NT, c1 = (long long)g.s[1].problems * g.s[1].upp * g.s[1].NT;
    const long long n0 = (long long)g.s[0].problems * g.s[0].upp;
    auto first = [&](long long c) {              // first unit (over both sides) whose start cost is >= c
      return c <= c0 ? (g.s[0].NT > 0 ? (c + g.s[0].NT - 1) / g.s[0].NT : 0) : n0 + (c - c0 + g.s[1].NT - 1) / g.s[1].NT;
    };
    const long long a = first((c0 + c1) * blockIdx.x / gridDim.x), b = first((c0 + c1) * (blockIdx.x + 1) / gridDim.x);
    left = b - a;
    side = a >= n0 ? 1 : 0;
    const long long k = a - (side ? n0 : 0);
    const int upp = g.s[side].upp > 0 ? g.s[side].upp : 1;
    prob = (int)(k / upp); u = (int)(k % upp);
  }
  __device__ __forceinline__ bool more() const { return left > 0; }
  // the current unit is this CTA's last of its problem
  __device__ __forceinline__ bool last(const Args& g) const { return left == 1 || u + 1 == g.s[side].upp; }
  // the next unit; true when it belongs to another problem
  __device__ __forceinline__ bool next(const Args& g) {
    --left;
    if (++u < g.s[side].upp) return false;
    u = 0;
    if (++prob == g.s[side].problems) { prob = 0; side = 1; }
    return true;
  }
};

// DIST: the units without a flagged point tile are passed over by every role
template <int R> __device__ __forceinline__ bool flagged(const Args& g, const Walk& w) {
  const Side& sd = g.s[w.side];
  const int tiles = (g.N + kRows - 1) / kRows;
  int f = 0;
  for (int r = 0; r < R; ++r) if (w.u * R + r < tiles) f |= sd.flags[(size_t)w.prob * tiles + w.u * R + r];
  return f != 0;
}

template <int D, int R, bool DIST>     // R: point tiles per unit; DIST: write |c|^2 - 2 x.c of the flagged tiles instead of the assignments
__global__ void __launch_bounds__(kThreads, 1)
k_assign_tc(const __grid_constant__ CUtensorMap tx0, const __grid_constant__ CUtensorMap th0, const __grid_constant__ CUtensorMap tl0,
            const __grid_constant__ CUtensorMap tx1, const __grid_constant__ CUtensorMap th1, const __grid_constant__ CUtensorMap tl1,
            const __grid_constant__ Args g, int* __restrict__ status) {
  extern __shared__ __align__(1024) unsigned char sm_raw[];
  __shared__ Bars bars;
  __shared__ uint32_t tbase_s;
  constexpr int G = D / 64, kX = kRows * D * 2, PPT = 2 * G;                     // pieces per centre tile: hi groups, lo groups
  unsigned char* sm = sm_raw + ((1024u - (tc::smem_u32(sm_raw) & 1023u)) & 1023u);
  unsigned char* Xs = sm;
  unsigned char* ring = sm + kXStages * kX;
  const int tid = threadIdx.x, warp = tc::warp_index(), ns = g.ns, N = g.N;
  if (warp == 0) tc::tmem_alloc(&tbase_s, 4 * kCols);
  if (tid == 0) {
    for (int s = 0; s < kXStages; ++s) { tc::mbar_init(&bars.xfull[s], 1); tc::mbar_init(&bars.xempty[s], 1); }
    for (int s = 0; s < ns; ++s) { tc::mbar_init(&bars.full[s], 1); tc::mbar_init(&bars.empty[s], 1); }
    for (int b = 0; b < 4; ++b) { tc::mbar_init(&bars.tfull[b >> 1][b & 1], 1); tc::mbar_init(&bars.tempty[b >> 1][b & 1], 128); }
    tc::mbar_init_fence();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tbase = tbase_s;
  bool ok = true;
  pdl_wait();
  pdl_trigger();
  Walk w(g);

  if (warp >= 8 && warp < 8 + kXProd) {
    if ((tid & 31) == 0) {                                 // ---- points: this thread takes every kXProd-th tile
      int turn = warp - 8;
      for (int s = 0, ph = 0; w.more() && ok; w.next(g)) {
        if (DIST && !flagged<R>(g, w)) continue;
        for (int r = 0; r < R; ++r) {
          if (turn == 0) {
            if (!tc::mbar_wait(&bars.xempty[s], ph ^ 1)) { ok = false; break; }
            tc::mbar_expect_tx(&bars.xfull[s], kX);
            // (a tile past the end of the points starts at the last row: its distances are never used)
            const int row = w.prob * N + min(N - 1, (w.u * R + r) * kRows);
#pragma unroll
            for (int q = 0; q < G; ++q) tc::tma_load_2d(Xs + s * kX + q * kRows * 128, w.side ? &tx1 : &tx0, 64 * q, row, &bars.xfull[s]);
          }
          turn = turn == 0 ? kXProd - 1 : turn - 1;
          if (++s == kXStages) { s = 0; ph ^= 1; }
        }
      }
    }
  } else if (warp >= 8 + kXProd && warp < 8 + kXProd + kCProd) {
    if ((tid & 31) == 0) {                                 // ---- centre pieces: this thread takes every kCProd-th piece
      int turn = warp - 8 - kXProd;
      bool fresh = true;
      for (int s = 0, ph = 0; w.more() && ok; fresh = w.next(g)) {
        const Side& sd = g.s[w.side];
        if (DIST && !flagged<R>(g, w)) continue;
        if (!DIST && sd.NT * PPT <= ns && !fresh) continue;         // resident
        for (int t = 0; t < sd.NT && ok; ++t)
#pragma unroll
          for (int p = 0; p < PPT; ++p) {
            if (turn == 0) {
              if (!tc::mbar_wait(&bars.empty[s], ph ^ 1)) { ok = false; break; }
              tc::mbar_expect_tx(&bars.full[s], kPiece);
              const void* map = p < G ? (w.side ? &th1 : &th0) : (w.side ? &tl1 : &tl0);
              tc::tma_load_2d(ring + s * kPiece, map, 64 * (p % G), w.prob * sd.C + t * kCols, &bars.full[s]);
            }
            turn = turn == 0 ? kCProd - 1 : turn - 1;
            if (++s == ns) { s = 0; ph ^= 1; }
          }
      }
    }
  } else if (warp == 8 + kXProd + kCProd) {                // ---- MMA issuer (whole warp, one elected lane)
    const uint32_t idesc = tc::idesc_bf16(kRows, kCols, 0, 0);
    const uint64_t dx0 = tc::smem_desc_sw128(tc::smem_u32(Xs), 16, 1024), dr0 = tc::smem_desc_sw128(tc::smem_u32(ring), 16, 1024);
    bool fresh = true;
    int s = 0, ph = 0, x = 0, xph = 0, b = 0, bph = 0;
    int s0 = 0;                                            // first ring slot of a resident problem
    while (w.more() && ok) {
      if (DIST && !flagged<R>(g, w)) { w.next(g); continue; }
      const int NT = g.s[w.side].NT;
      const bool res = !DIST && NT * PPT <= ns;            // (with units passed over, a problem's first and last are not known)
      uint64_t dx[R];
      int xs[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (!tc::mbar_wait(&bars.xfull[x], xph)) ok = false;
        xs[r] = x;
        dx[r] = tc::desc_step(dx0, (uint32_t)x * kX);
        if (++x == kXStages) { x = 0; xph ^= 1; }
      }
      if (res && fresh) s0 = s;
      int rs = s0;                                         // slot walked by a resident problem's later units
      const bool last_of_problem = w.last(g);
      for (int t = 0; t < NT && ok; ++t) {
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (!tc::mbar_wait(&bars.tempty[r][b], bph ^ 1)) ok = false;
        tc::fence_after_sync();
#pragma unroll
        for (int p = 0; p < PPT; ++p) {
          const int slot = res && !fresh ? rs : s;
          if (!res || fresh) {
            if (!tc::mbar_wait(&bars.full[s], ph)) ok = false;
            if (++s == ns) { s = 0; ph ^= 1; }
          }
          if (!ok) break;
          tc::fence_after_sync();
          const uint64_t dc = tc::desc_step(dr0, (uint32_t)slot * kPiece);
#pragma unroll
          for (int r = 0; r < R; ++r)
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
              tc::mma_bf16_ss_warp(tbase + (r * 2 + b) * kCols, tc::desc_step(dx[r], (p % G) * kRows * 128 + ks * 32), tc::desc_step(dc, ks * 32),
                                   idesc, (p | ks) != 0);
          if (!res || last_of_problem) tc::mma_commit_warp(&bars.empty[slot]);   // the piece may be overwritten
          if (++rs == ns) rs = 0;
        }
        if (!ok) break;
#pragma unroll
        for (int r = 0; r < R; ++r) tc::mma_commit_warp(&bars.tfull[r][b]);
        b ^= 1; bph ^= b == 0;
      }
#pragma unroll
      for (int r = 0; r < R; ++r) tc::mma_commit_warp(&bars.xempty[xs[r]]);
      fresh = w.next(g);
    }
  } else if ((warp >> 2) < R) {
    // ---- arg-min sweep: thread = point row
    const int row = tid & 127, r = warp >> 2;
    const uint32_t tlane = tbase + ((uint32_t)((warp & 3) * 32) << 16) + r * 2 * kCols;
    for (int b = 0, bph = 0; w.more() && ok; w.next(g)) {
      if (DIST && !flagged<R>(g, w)) continue;
      const Side& sd = g.s[w.side];
      const int C = sd.C, at = (w.u * R + r) * kRows + row;
      const float* cn = sd.cnorm + (size_t)w.prob * sd.NT * kCols;
      // four running minima per row (columns mod 4) instead of one chain of 128 dependent compare-and-selects per tile
      float best[4];
      int bidx[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) { best[e] = INFINITY; bidx[e] = 0x7fffffff; }
      for (int t = 0; t < sd.NT; ++t) {
        if (!tc::mbar_wait(&bars.tfull[r][b], bph)) { ok = false; break; }
        tc::fence_after_sync();
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float v[32];
          float4 nn[8];
          const int c0 = t * kCols + 32 * q;
#pragma unroll
          for (int k = 0; k < 8; ++k) nn[k] = *reinterpret_cast<const float4*>(cn + c0 + 4 * k);
          tc::tmem_ld32(tlane + b * kCols + 32 * q, v);
          if (q == 3) { tc::fence_before_sync(); tc::mbar_arrive(&bars.tempty[r][b]); }
#pragma unroll
          for (int k = 0; k < 32; k += 4) {
            const float4 n4 = nn[k / 4];
            v[k] = fmaf(-2.f, v[k], n4.x); v[k + 1] = fmaf(-2.f, v[k + 1], n4.y);
            v[k + 2] = fmaf(-2.f, v[k + 2], n4.z); v[k + 3] = fmaf(-2.f, v[k + 3], n4.w);
#pragma unroll
            for (int e = 0; e < 4; ++e)
              if (!DIST) argmin_step(v[k + e], c0 + k + e, best[e], bidx[e]);      // ascending index: ties keep the lower
          }
          if (DIST && at < N) {
            float* dr = sd.dist + ((size_t)w.prob * N + at) * C + c0;
            if (c0 + 32 <= C && (C & 3) == 0) {
#pragma unroll
              for (int k = 0; k < 32; k += 4) *reinterpret_cast<float4*>(dr + k) = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
            } else {
#pragma unroll
              for (int k = 0; k < 32; ++k) if (c0 + k < C) dr[k] = v[k];
            }
          }
        }
        b ^= 1; bph ^= b == 0;
      }
#pragma unroll
      for (int e = 1; e < 4; ++e) argmin_tie_step(best[e], bidx[e], best[0], bidx[0]);
      // a row of NaN or infinities never compares below the running minimum: it goes to cluster 0
      if (!DIST && ok && at < N) sd.assign[(size_t)w.prob * N + at] = (unsigned)bidx[0] < (unsigned)C ? bidx[0] : 0;
    }
  }
  if (!ok) report_status(status, MUSE_STATUS_ASSIGN_TIMEOUT);
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tbase, 4 * kCols);
}

}  // namespace at

int assign_tc(const LloydSide* sides, int nsides, int N, int D, int distances, int* status, cudaStream_t st) {
  at::Args g = {};
  CUtensorMap m[6];
  const bool dist = distances != 0;
  const int sms = sm_count();
  long long tiles = 0;
  for (int k = 0; k < nsides; ++k) tiles += (long long)sides[k].problems * cdiv(N, at::kRows);
  g.N = N;
  const int R = tiles >= 2 * sms ? 2 : 1;                          // two-tile units once every SM gets one
  g.ns = D == 128 ? 5 : 9;
  long long units = 0;
  for (int k = 0; k < 2; ++k) {
    const LloydSide& s = sides[k < nsides ? k : 0];         // (a missing side has no units; its maps are never used)
    MUSE_RC(make_tmap_bf16_rows(&m[3 * k], s.X, (uint64_t)s.problems * N, (uint32_t)D, at::kRows));
    MUSE_RC(make_tmap_bf16_rows(&m[3 * k + 1], s.chi, (uint64_t)s.problems * s.C, (uint32_t)D, at::kCols));
    MUSE_RC(make_tmap_bf16_rows(&m[3 * k + 2], s.clo, (uint64_t)s.problems * s.C, (uint32_t)D, at::kCols));
    g.s[k] = at::Side{s.cnorm, s.assign, s.dist, s.flags, k < nsides ? s.problems : 0, s.C, cdiv(s.C, at::kCols), cdiv(N, at::kRows * R)};
    units += (long long)g.s[k].problems * g.s[k].upp;
  }
  const int grid = units < sms ? (int)units : sms;
  const size_t smem = (size_t)at::kXStages * at::kRows * D * 2 + (size_t)g.ns * at::kPiece + 1024;
  prof_mark("k_assign_tc", st);
#define MUSE_AT_LAUNCH(DD, RR, DI) return launch_pdl(at::k_assign_tc<DD, RR, DI>, dim3(grid), at::kThreads, smem, st, m[0], m[1], m[2], m[3], m[4], m[5], g, status)
#define MUSE_AT_D(DD)                                                     \
  {                                                                       \
    if (R == 2) { if (dist) MUSE_AT_LAUNCH(DD, 2, true); MUSE_AT_LAUNCH(DD, 2, false); } \
    if (dist) MUSE_AT_LAUNCH(DD, 1, true);                                \
    MUSE_AT_LAUNCH(DD, 1, false);                                         \
  }
  if (D == 128) MUSE_AT_D(128)
  MUSE_AT_D(64)
#undef MUSE_AT_D
#undef MUSE_AT_LAUNCH
}

}  // namespace muse
