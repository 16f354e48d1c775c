// Clustering stage: Lloyd k-means (Appendix "Clustering Details").  The query side and the key side are independent
// problems of the same shape of work, so every kernel takes both in one launch: an iteration is three launches
// (assignment, bucket_sort, k_update); small problems take all iterations in one (lloyd_small.cu).
#include "common.cuh"
#include "feistel.cuh"

namespace muse {

struct LloydSides { LloydSide s[2]; int N, S; };

// the side and the problem-and-centre index of flat centre index e over both sides
__device__ __forceinline__ const LloydSide& side_of_centre(const LloydSides& g, long long& e) {
  const long long n0 = (long long)g.s[0].problems * g.s[0].C;
  if (e < n0) return g.s[0];
  e -= n0;
  return g.s[1];
}
__device__ __forceinline__ size_t cnorm_index(int prob, int c, int C) { return (size_t)prob * (cdiv(C, kAsgTile) * kAsgTile) + c; }

// bf16 hi + lo planes of a centre's element (the operands of the tensor-core assignment)
__device__ __forceinline__ void split_centre(const LloydSide& sd, size_t e, float x) {
  const __nv_bfloat16 h = __float2bfloat16_rn(x);
  ((__nv_bfloat16*)sd.chi)[e] = h;
  ((__nv_bfloat16*)sd.clo)[e] = __float2bfloat16_rn(x - __bfloat162float(h));
}

// Start centres (drawn by index, by the seeded stride, or the caller's), their squared norms and bf16 planes: a warp
// per centre.  The padding of cnorm is set to infinity here, once per call.
template <class T>
__global__ void __launch_bounds__(256)
k_init_centres(const __grid_constant__ LloydSides g, int D, int init_mode, uint64_t seed, int32_t* __restrict__ clear) {
  const int lane = threadIdx.x & 31;
  long long e = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  pdl_wait();
  pdl_trigger();
  if (clear != nullptr && blockIdx.x == 0 && threadIdx.x < kStatusWords) clear[threadIdx.x] = 0;
  const LloydSide& sd = side_of_centre(g, e);
  if (e >= (long long)sd.problems * sd.C) return;
  const int prob = (int)(e / sd.C), c = (int)(e % sd.C);
  float* o = sd.centres + (size_t)e * D;
  float s = 0.f;
  if (init_mode != MUSE_INIT_CENTRES) {
    int idx;
    if (init_mode == MUSE_INIT_INDICES) idx = sd.init_idx[e];
    else idx = feistel_permute(c * (g.N / sd.C), g.N, seed, (uint64_t)prob * 2 + sd.kind);
    idx = min(max(idx, 0), g.N - 1);
    const T* x = (const T*)sd.X + ((size_t)prob * g.N + idx) * D;
    for (int d = lane; d < D; d += 32) {
      const float v = to_f(x[d]);
      o[d] = v;
      s = fmaf(v, v, s);
      if (sizeof(T) == 2) split_centre(sd, (size_t)e * D + d, v);
    }
  } else {
    for (int d = lane; d < D; d += 32) {
      const float v = o[d];
      s = fmaf(v, v, s);
      if (sizeof(T) == 2) split_centre(sd, (size_t)e * D + d, v);
    }
  }
  s = warp_sum(s);
  if (lane == 0) sd.cnorm[cnorm_index(prob, c, sd.C)] = s;
  if (c == sd.C - 1)
    for (int k = sd.C + lane; k < cdiv(sd.C, kAsgTile) * kAsgTile; k += 32) sd.cnorm[cnorm_index(prob, k, sd.C)] = INFINITY;
}

// Assignment for fp32 inputs: argmin_c |c|^2 - 2 x.c, fp32 FFMA, 16 * RPT points x 16 * CPT centres per tile, RPT x CPT
// per thread.  The small tiles serve small problems, where 128-point tiles leave most of the chip idle and 64-centre
// tiles multiply zeros (1024 points, 8 and 16 centres: 14.4 us per side -> 8 us for both).
constexpr int kAsgThreads = 256;

template <int D, int RPT, int CPT>
__global__ void __launch_bounds__(kAsgThreads)
k_assign(const __grid_constant__ LloydSides g, int distances) {
  constexpr int LD = D + 4, ROWS = 16 * RPT, COLS = 16 * CPT;
  extern __shared__ float smf[];
  float* Xs = smf;                       // [ROWS][LD]
  float* Cs = Xs + ROWS * LD;            // [COLS][LD]
  float* cn = Cs + COLS * LD;            // [COLS]
  const int N = g.N;
  int prob = blockIdx.y;
  const bool second = prob >= g.s[0].problems;
  const LloydSide& sd = g.s[second ? 1 : 0];
  if (second) prob -= g.s[0].problems;
  const int C = sd.C, row0 = blockIdx.x * ROWS;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  pdl_wait();
  pdl_trigger();
  const float* Xp = (const float*)sd.X + (size_t)prob * N * D;
  const float* Cp = sd.centres + (size_t)prob * C * D;
  const float* cnp = sd.cnorm + cnorm_index(prob, 0, C);
  if (distances && sd.flags[(size_t)prob * cdiv(N, kAsgTile) + row0 / kAsgTile] == 0) return;
  float* dist_out = distances ? sd.dist : nullptr;
  for (int e = tid; e < ROWS * (D / 4); e += kAsgThreads) {
    int r = e / (D / 4), q = e % (D / 4);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row0 + r < N) v = ld4(Xp + (size_t)(row0 + r) * D + q * 4);
    st4(Xs + r * LD + q * 4, v);
  }
  float best[RPT]; int bidx[RPT];
#pragma unroll
  for (int r = 0; r < RPT; ++r) { best[r] = INFINITY; bidx[r] = 0x7fffffff; }
  for (int c0 = 0; c0 < C; c0 += COLS) {
    __syncthreads();
    for (int e = tid; e < COLS * (D / 4); e += kAsgThreads) {
      int r = e / (D / 4), q = e % (D / 4);
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (c0 + r < C) v = ld4(Cp + (size_t)(c0 + r) * D + q * 4);
      st4(Cs + r * LD + q * 4, v);
    }
    if (tid < COLS) cn[tid] = (c0 + tid < C) ? cnp[c0 + tid] : INFINITY;
    __syncthreads();
    float acc[RPT][CPT];
#pragma unroll
    for (int r = 0; r < RPT; ++r)
#pragma unroll
      for (int k = 0; k < CPT; ++k) acc[r][k] = 0.f;
#pragma unroll 4
    for (int d = 0; d < D; d += 4) {
      float4 cv[CPT];
#pragma unroll
      for (int k = 0; k < CPT; ++k) cv[k] = ld4(Cs + (tx * CPT + k) * LD + d);
#pragma unroll
      for (int r = 0; r < RPT; ++r) {
        float4 xv = ld4(Xs + (ty * RPT + r) * LD + d);
#pragma unroll
        for (int k = 0; k < CPT; ++k) {
          acc[r][k] = fmaf(xv.x, cv[k].x, acc[r][k]);
          acc[r][k] = fmaf(xv.y, cv[k].y, acc[r][k]);
          acc[r][k] = fmaf(xv.z, cv[k].z, acc[r][k]);
          acc[r][k] = fmaf(xv.w, cv[k].w, acc[r][k]);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < RPT; ++r)
#pragma unroll
      for (int k = 0; k < CPT; ++k) {
        float dist = fmaf(-2.f, acc[r][k], cn[tx * CPT + k]);
        int c = c0 + tx * CPT + k;
        if (dist < best[r]) { best[r] = dist; bidx[r] = c; }   // ascending c: ties keep the lower
        // (optional output: the whole matrix |c|^2 - 2 x.c, for the balanced assignment's second step)
        if (dist_out != nullptr && c < C && row0 + ty * RPT + r < N) dist_out[((size_t)prob * N + row0 + ty * RPT + r) * C + c] = dist;
      }
  }
#pragma unroll
  for (int r = 0; r < RPT; ++r) {
    float b = best[r]; int i = bidx[r];
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
      float ob = __shfl_xor_sync(0xffffffffu, b, o);
      int oi = __shfl_xor_sync(0xffffffffu, i, o);
      if (ob < b || (ob == b && oi < i)) { b = ob; i = oi; }
    }
    int row = row0 + ty * RPT + r;
    // a row of NaN or infinities never compares below the running minimum: it goes to cluster 0
    if (tx == 0 && row < N) sd.assign[(size_t)prob * N + row] = (unsigned)i < (unsigned)C ? i : 0;
  }
}

template <int D, int RPT, int CPT>
static int assign_f32_v(const LloydSides& g, int nprob, int distances, cudaStream_t st) {
  const size_t smem = (size_t)((16 * RPT + 16 * CPT) * (D + 4) + 16 * CPT) * sizeof(float);
  return launch_pdl(k_assign<D, RPT, CPT>, dim3(cdiv(g.N, 16 * RPT), nprob), kAsgThreads, smem, st, g, distances);
}

template <int D>
static int assign_f32(const LloydSides& g, int nsides, int distances, cudaStream_t st) {
  int nprob = 0, C = 0;
  for (int k = 0; k < nsides; ++k) { nprob += g.s[k].problems; C = C > g.s[k].C ? C : g.s[k].C; }
  prof_mark("k_assign", st);
  if ((long long)nprob * cdiv(g.N, 128) >= 2 * sm_count()) return assign_f32_v<D, 8, 4>(g, nprob, distances, st);   // two rounds of full tiles
  if (C > 16) return assign_f32_v<D, 2, 4>(g, nprob, distances, st);
  return assign_f32_v<D, 2, 1>(g, nprob, distances, st);
}

// Centre update: mean of the members, summed with a fixed reduction tree (slot s of the CTA adds members
// s, s + SLOTS, ... in bucket order, then the slots are added in order), so the result does not depend
// on scheduling.  An empty cluster keeps its centre.  One 256-thread CTA per cluster; a lane owns 16 bytes
// of a row, and every slot keeps four row loads in flight (the member list is an indirection, so a
// single load per slot leaves the kernel waiting on memory latency).
constexpr int kUpdThreads = 256;

__device__ __forceinline__ void ld16f(const float* p, float (&x)[4]) { const float4 v = *reinterpret_cast<const float4*>(p); x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w; }
__device__ __forceinline__ void ld16f(const __nv_bfloat16* p, float (&x)[8]) {
  const uint4 u = *reinterpret_cast<const uint4*>(p);
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) { x[2 * k] = __uint_as_float(w[k] << 16); x[2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u); }
}

template <class T, int D>
__global__ void __launch_bounds__(kUpdThreads)
k_update(const __grid_constant__ LloydSides g) {
  constexpr int VEC = 16 / (int)sizeof(T);     // elements per lane
  constexpr int LPR = D / VEC;                 // lanes per row
  constexpr int RPW = 32 / LPR;                // rows per warp step
  constexpr int SLOTS = (kUpdThreads / 32) * RPW;
  __shared__ float part[SLOTS][D];
  __shared__ float n2_s[kUpdThreads / 32];
  long long e = blockIdx.x;
  const LloydSide& sd = side_of_centre(g, e);
  const int N = g.N, S = g.S, C = sd.C, kind = sd.kind, prob = (int)(e / C), c = (int)(e % C);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sub = lane / LPR, q = lane % LPR;
  const int slot = warp * RPW + sub;
  const T* Xp = (const T*)sd.X + (size_t)prob * N * D + q * VEC;
  const int32_t* o = sd.off + (size_t)prob * (C * S + 1);
  const int32_t* pm = sd.perm + (size_t)prob * N;
  pdl_wait();
  pdl_trigger();
  float s[VEC];
#pragma unroll
  for (int k = 0; k < VEC; ++k) s[k] = 0.f;
  int count = 0;
  const int nranges = kind == 0 ? S : 1;
  for (int r = 0; r < nranges; ++r) {
    const int p0 = kind == 0 ? o[r * C + c] : o[c * S];
    const int p1 = kind == 0 ? o[r * C + c + 1] : o[(c + 1) * S];
    count += p1 - p0;
    for (int p = p0 + slot; p < p1; p += 4 * SLOTS) {
      int idx[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        idx[u] = p + u * SLOTS < p1 && MUSE_IN_RANGE(p + u * SLOTS, N) ? pm[p + u * SLOTS] : -1;
        if (idx[u] >= 0 && !MUSE_IN_RANGE(idx[u], N)) idx[u] = -1;
      }
      float v[4][VEC];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (idx[u] >= 0) ld16f(Xp + (size_t)idx[u] * D, v[u]);
        else {
#pragma unroll
          for (int k = 0; k < VEC; ++k) v[u][k] = 0.f;
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int k = 0; k < VEC; ++k) s[k] += v[u][k];
    }
  }
#pragma unroll
  for (int k = 0; k < VEC; ++k) part[slot][q * VEC + k] = s[k];
  __syncthreads();
  float n2 = 0.f;
  if (threadIdx.x < D) {
    const int d = threadIdx.x;
    float tot = 0.f;
    float* dst = sd.centres + (size_t)e * D + d;
#pragma unroll
    for (int k = 0; k < SLOTS; ++k) tot += part[k][d];
    if (count > 0) { tot *= 1.f / (float)count; *dst = tot; }
    else tot = *dst;
    if (sizeof(T) == 2) split_centre(sd, (size_t)e * D + d, tot);
    n2 = tot * tot;
  }
  n2 = warp_sum(n2);
  if (lane == 0) n2_s[warp] = n2;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
#pragma unroll
    for (int k = 0; k < D / 32; ++k) t += n2_s[k];
    sd.cnorm[cnorm_index(prob, c, C)] = t;
  }
}

template <class T, int D>
static int lloyd_t(LloydSides& g, const Dims& d, int nsides, int init_mode, uint64_t seed, int T_iters, bool fresh, int* status, cudaStream_t st) {
  // the status words are cleared by the first kernel of the call (k-means++ reports into them, so before it by a memset)
  int32_t* clear = fresh ? status : nullptr;
  if (init_mode == MUSE_INIT_KMEANSPP) {
    if (fresh) MUSE_CUDA_OK(cudaMemsetAsync(status, 0, kStatusWords * sizeof(int32_t), st));
    clear = nullptr;
    // the draws borrow two arrays that the iterations only fill later: perm as the running minimum distance
    // [problems, N] fp32, off (at least C + 1 words per problem) as the drawn indices [problems, C]
    KmeansppSide pp[2];
    for (int k = 0; k < nsides; ++k) {
      LloydSide& s = g.s[k];
      pp[k] = KmeansppSide{s.X, reinterpret_cast<float*>(s.perm), s.off, s.problems, s.C, s.kind};
      s.init_idx = s.off;
    }
    MUSE_RC(kmeanspp(sizeof(T) == 2 ? MUSE_BF16 : MUSE_F32, pp, nsides, d.N, D, seed, status, st));
    init_mode = MUSE_INIT_INDICES;
  }
  long long centres = 0;
  SortSide sort[2];
  for (int k = 0; k < nsides; ++k) {
    const LloydSide& s = g.s[k];
    centres += (long long)s.problems * s.C;
    sort[k] = SortSide{s.assign, s.off, s.perm, s.problems, s.C, s.kind};
  }
  prof_mark("k_init_centres", st);
  MUSE_RC(launch_pdl(k_init_centres<T>, dim3((unsigned)((centres + 7) / 8)), 256, 0, st, g, D, init_mode, seed, clear));
  bool taken = false;
  MUSE_RC(lloyd_small(d, sizeof(T) == 2 ? MUSE_BF16 : MUSE_F32, g.s, nsides, T_iters, &taken, status, st));
  if (taken) return MUSE_OK;
  for (int it = 0; it <= T_iters; ++it) {
    const bool last = it == T_iters;
    if (sizeof(T) == 2) {                      // bf16 inputs: distances on the tensor cores
      MUSE_RC(assign_tc(g.s, nsides, d.N, D, 0, status, st));
    } else {
      MUSE_RC(assign_f32<D>(g, nsides, 0, st));
    }
    if (last) break;
    MUSE_RC(bucket_sort(sort, nsides, d.N, d.S, d.Bs, st));
    prof_mark("k_update", st);
    MUSE_RC(launch_pdl(k_update<T, D>, dim3((unsigned)centres), kUpdThreads, 0, st, g));
  }
  return MUSE_OK;
}

int assign_distances(const Dims& d, int dtype, const LloydSide& side, int* status, cudaStream_t st) {
  if (dtype == MUSE_BF16) return assign_tc(&side, 1, d.N, d.D, 1, status, st);
  LloydSides g = {};
  g.s[0] = side;
  g.N = d.N; g.S = d.S;
  return d.D == 64 ? assign_f32<64>(g, 1, 1, st) : assign_f32<128>(g, 1, 1, st);
}

void lloyd_side_ws(const Dims& d, Arena& ar, LloydSide& s) {
  const size_t P = (size_t)s.problems;
  s.cnorm = ar.take<float>(P * cdiv(s.C, kAsgTile) * kAsgTile);
  s.off = ar.take<int32_t>(P * ((size_t)s.C * d.S + 1));
  s.perm = ar.take<int32_t>(P * d.N);
  s.chi = ar.take<__nv_bfloat16>(P * s.C * d.D);
  s.clo = ar.take<__nv_bfloat16>(P * s.C * d.D);
}

size_t lloyd_ws_bytes(const Dims& d, int problems, int C) {
  Arena ar(nullptr);
  LloydSide s = {};
  s.problems = problems; s.C = C;
  lloyd_side_ws(d, ar, s);
  return ar.used;
}

int lloyd(const Dims& d, int dtype, LloydSide* sides, int nsides, int init_mode, uint64_t seed, int T, bool clear, int* status, cudaStream_t st) {
  LloydSides g = {};
  for (int k = 0; k < nsides; ++k) g.s[k] = sides[k];
  g.N = d.N; g.S = d.S;
  if (dtype == MUSE_F32)
    return d.D == 64 ? lloyd_t<float, 64>(g, d, nsides, init_mode, seed, T, clear, status, st)
                     : lloyd_t<float, 128>(g, d, nsides, init_mode, seed, T, clear, status, st);
  return d.D == 64 ? lloyd_t<__nv_bfloat16, 64>(g, d, nsides, init_mode, seed, T, clear, status, st)
                   : lloyd_t<__nv_bfloat16, 128>(g, d, nsides, init_mode, seed, T, clear, status, st);
}

}  // namespace muse
