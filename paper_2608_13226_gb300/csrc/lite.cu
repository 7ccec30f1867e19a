// K6-K8: CoverPrune-Lite (Sec. 4.1, Eqs. lite_group, lite_select; Sec. 4.2,
// Eqs. blk_plan, blk_ot).
#include "common.cuh"
#include "bf16_dot.cuh"

namespace cp {

// Spread the low 10 bits of q so that bit i lands on bit 3i.
__device__ __forceinline__ uint32_t spread3(uint32_t q) {
  q &= 0x3FFu;
  q = (q | (q << 16)) & 0x030000FFu;
  q = (q | (q << 8)) & 0x0300F00Fu;
  q = (q | (q << 4)) & 0x030C30C3u;
  q = (q | (q << 2)) & 0x09249249u;
  return q;
}

// Voxel cell of one coordinate: floor((x - lo) / voxel) in fp32 with each
// operation rounded once, clamped to [0, 1023].
__device__ __forceinline__ uint32_t voxel_cell(float x, float lo, float voxel) {
  float cell = floorf(__fdiv_rn(__fsub_rn(x, lo), voxel));
  cell = fminf(fmaxf(cell, 0.0f), 1023.0f);
  return (uint32_t)cell;
}

// K6: Morton code per token and the order by (code, index).  One block per
// scene: a stable radix sort of the codes in shared memory, 8 bits a pass, as
// many passes as the largest code has (a 8 m room at 0.2 m: 18 bits, 3).  Each
// warp takes a contiguous run of tokens: it counts its digits, the counts are
// scanned (digit by digit, warp by warp), and it moves its tokens, 32 at a
// time in order.  Bound by those chains of shared-memory latencies; 16384
// tokens 64 us, the bitonic sort of 64-bit keys before took 165.
constexpr int MT_WARPS = 32, MT_BINS = 256;

__global__ void __launch_bounds__(32 * MT_WARPS) k_morton(const float* __restrict__ pos_all,
                                                          const SceneStats* __restrict__ stats,
                                                          float voxel, int N, int Np,
                                                          int32_t* __restrict__ perm_all) {
  extern __shared__ __align__(16) unsigned char mt_smem[];
  uint32_t* K = reinterpret_cast<uint32_t*>(mt_smem);  // [Np] codes, and [Np] for the next pass
  uint32_t* K2 = K + Np;
  uint16_t* I = reinterpret_cast<uint16_t*>(K2 + Np);  // [Np] tokens, and [Np]
  uint16_t* I2 = I + Np;
  uint16_t* hist = I2 + Np;  // [MT_WARPS][MT_BINS] counts, then places
  __shared__ uint32_t s_part[4][MT_BINS];
  __shared__ uint32_t s_base[MT_BINS];
  __shared__ uint32_t s_w[8];
  __shared__ uint32_t s_max;
  const int b = blockIdx.x, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float* X = pos_all + (size_t)b * N * 3;
  const float lx = stats[b].bbox_min[0], ly = stats[b].bbox_min[1], lz = stats[b].bbox_min[2];
  if (threadIdx.x == 0) s_max = 0u;
  __syncthreads();
  uint32_t top = 0u;
#pragma unroll 4
  for (int j = threadIdx.x; j < N; j += 32 * MT_WARPS) {
    const uint32_t code = spread3(voxel_cell(X[3 * j], lx, voxel)) |
                          (spread3(voxel_cell(X[3 * j + 1], ly, voxel)) << 1) |
                          (spread3(voxel_cell(X[3 * j + 2], lz, voxel)) << 2);
    K[j] = code;
    I[j] = (uint16_t)j;
    top = max(top, code);
  }
  top = __reduce_max_sync(0xFFFFFFFFu, top);
  if (lane == 0) atomicMax(&s_max, top);
  __syncthreads();
  const int bits = 32 - __clz((int)s_max);
  const int per = ((N + MT_WARPS - 1) / MT_WARPS + 31) & ~31;
  const int j0 = min(N, w * per), j1 = min(N, j0 + per);
  const uint32_t lt = (1u << lane) - 1u;
  uint16_t* mine = hist + w * MT_BINS;
  for (int sh = 0; sh < bits; sh += 8) {
    for (int d = lane; d < MT_BINS; d += 32) mine[d] = 0;
    __syncwarp();
    for (int j = j0; j < j1; j += 32) {
      const bool in = j + lane < j1;
      const uint32_t act = __ballot_sync(0xFFFFFFFFu, in);
      if (in) {
        const uint32_t d = (K[j + lane] >> sh) & 255u;
        const uint32_t same = __match_any_sync(act, d);
        if ((same & lt) == 0u) mine[d] += (uint16_t)__popc(same);
      }
      __syncwarp();
    }
    __syncthreads();
    {  // places: digits ascending, within a digit the warps ascending
      const int d = threadIdx.x & 255, q = threadIdx.x >> 8;
      uint32_t sum = 0u;
#pragma unroll
      for (int i = 0; i < 8; ++i) sum += hist[(8 * q + i) * MT_BINS + d];
      s_part[q][d] = sum;
      __syncthreads();
      uint32_t tot = 0u, incl = 0u;
      if (threadIdx.x < MT_BINS) {
        tot = s_part[0][d] + s_part[1][d] + s_part[2][d] + s_part[3][d];
        incl = tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
          if (lane >= o) incl += t;
        }
        if (lane == 31) s_w[w] = incl;
      }
      __syncthreads();
      if (threadIdx.x < MT_BINS)
        s_base[d] = incl - tot + __reduce_add_sync(0xFFFFFFFFu, lane < w ? s_w[lane & 7] : 0u);
      __syncthreads();
      uint32_t run = s_base[d];
      for (int i = 0; i < q; ++i) run += s_part[i][d];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const uint32_t c = hist[(8 * q + i) * MT_BINS + d];
        hist[(8 * q + i) * MT_BINS + d] = (uint16_t)run;
        run += c;
      }
      __syncthreads();
    }
    for (int j = j0; j < j1; j += 32) {
      const bool in = j + lane < j1;
      const uint32_t act = __ballot_sync(0xFFFFFFFFu, in);
      uint32_t k = 0u, d = 0u, same = 0u;
      int at = 0;
      if (in) {
        k = K[j + lane];
        d = (k >> sh) & 255u;
        same = __match_any_sync(act, d);
        at = (int)mine[d] + __popc(same & lt);
      }
      __syncwarp();
      if (in) {
        if ((same & lt) == 0u) mine[d] += (uint16_t)__popc(same);
        K2[at] = k;
        I2[at] = I[j + lane];
      }
      __syncwarp();
    }
    __syncthreads();
    uint32_t* tk = K;
    K = K2;
    K2 = tk;
    uint16_t* ti = I;
    I = I2;
    I2 = ti;
  }
  for (int p = threadIdx.x; p < N; p += 32 * MT_WARPS) perm_all[(size_t)b * N + p] = (int32_t)I[p];
}

int launch_morton(const float* pos, const SceneStats* stats, const DevParams& P, int64_t B, int64_t N,
                  int32_t* perm, cudaStream_t s) {
  const int Np = (int)((N + 7) & ~(int64_t)7);
  const size_t smem = 12 * (size_t)Np + sizeof(uint16_t) * MT_WARPS * MT_BINS;
  CP_TRY_STATUS(allow_smem((const void*)k_morton, smem, "launch_morton: smem attribute"));
  k_morton<<<(unsigned)B, 32 * MT_WARPS, smem, s>>>(pos, stats, P.voxel, (int)N, Np, perm);
  return last_launch_status();
}

// Block-wide inclusive scan over blockDim.x == 1024 values.
__device__ __forceinline__ int block_incl_max_int(int x, int* s_w, int* total) {
  const int l = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (l >= o) x = max(x, y);
  }
  if (l == 31) s_w[w] = x;
  __syncthreads();
  if (w == 0) {
    int y = s_w[l];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int z = __shfl_up_sync(0xFFFFFFFFu, y, o);
      if (l >= o) y = max(y, z);
    }
    s_w[l] = y;
  }
  __syncthreads();
  const int r = w > 0 ? max(x, s_w[w - 1]) : x;
  *total = s_w[31];
  __syncthreads();
  return r;
}

// K7: capacity-guided grouping of Eq. lite_group in exact integers.
//   Q_j = rint(v_j 2^40); P(p) = inclusive running mass in Morton order;
//   ideal start of group q >= 1: 1 + min{p : P(p) K >= q P(N-1)};
//   b_q = q + min(N - K, max_{q' <= q} (ideal_q' - q')), b_0 = 0, b_K = N.
// One block of 1024 threads per scene.  Each warp sums a contiguous run of the
// order, kept in shared memory; a group's start is searched there (all
// products fit 64 bits: P(N-1) is 2^40 and a little, K at most 2^14).
// Latency-bound: 16384 tokens 16 us; with the masses in global memory, a
// block scan per 1024 tokens and 128-bit products 43.
__global__ void __launch_bounds__(1024) k_groups(const float* __restrict__ v_all,
                                                 const int32_t* __restrict__ perm_all, int N, int K,
                                                 int32_t* __restrict__ gs_all) {
  extern __shared__ unsigned long long s_P[];  // [N] masses within a warp's run, inclusive
  __shared__ unsigned long long s_off[33];     // mass before each warp's run; [32]: all of it
  __shared__ int s_wi[32];
  const int b = blockIdx.x, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float* v = v_all + (size_t)b * N;
  const int32_t* perm = perm_all + (size_t)b * N;
  int32_t* gs = gs_all + (size_t)b * (K + 1);
  const int run = ((N + 31) / 32 + 31) & ~31;  // tokens a warp
  const int p0 = min(N, w * run), p1 = min(N, p0 + run);
  unsigned long long carry = 0ull;
  for (int p = p0; p < p1; p += 128) {  // four chunks' loads in flight
    float x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = p + 32 * u + lane;
      x[u] = i < p1 ? v[perm[i]] : 0.0f;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      // rint(v 2^40), the product exact
      unsigned long long q = x[u] > 0.0f ? __float2ull_rn(x[u] * 1099511627776.0f) : 0ull;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long t = __shfl_up_sync(0xFFFFFFFFu, q, o);
        if (lane >= o) q += t;
      }
      q += carry;
      carry = __shfl_sync(0xFFFFFFFFu, q, 31);
      const int i = p + 32 * u + lane;
      if (i < p1) s_P[i] = q;
    }
  }
  if (lane == 0) s_off[w] = carry;
  __syncthreads();
  if (w == 0) {
    unsigned long long q = s_off[lane];
    const unsigned long long own = q;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long t = __shfl_up_sync(0xFFFFFFFFu, q, o);
      if (lane >= o) q += t;
    }
    s_off[lane] = q - own;
    if (lane == 31) s_off[32] = q;
  }
  __syncthreads();
  const unsigned long long total = s_off[32];
  // ideal_q - q for q = 1..K-1, staged in gs[q]
  for (int q = 1 + threadIdx.x; q < K; q += 1024) {
    const unsigned long long target = (unsigned long long)q * total;
    // smallest p with P(p) K >= target (exists: P(N-1) K >= target): the run
    // first, then within it
    int r = 0;
    while (r < 31 && (r + 1) * run < N && s_off[r + 1] * (unsigned)K < target) ++r;
    const unsigned long long before = s_off[r];
    int lo = r * run, hi = min(N, lo + run) - 1;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if ((before + s_P[mid]) * (unsigned)K >= target) hi = mid; else lo = mid + 1;
    }
    gs[q] = (lo + 1) - q;
  }
  __syncthreads();
  int top = INT32_MIN;
  for (int c0 = 1; c0 < K; c0 += 1024) {
    const int q = c0 + threadIdx.x;
    const int x = q < K ? gs[q] : INT32_MIN;
    int tot;
    const int m = max(top, block_incl_max_int(x, s_wi, &tot));
    if (q < K) gs[q] = q + min(N - K, m);
    top = max(top, tot);
  }
  if (threadIdx.x == 0) {
    gs[0] = 0;
    gs[K] = N;
  }
}

int launch_groups(const float* v, const int32_t* perm, int64_t B, int64_t N, int64_t K,
                  int32_t* gs, cudaStream_t s) {
  const size_t smem = sizeof(unsigned long long) * (size_t)N;
  CP_TRY_STATUS(allow_smem((const void*)k_groups, smem, "launch_groups: smem attribute"));
  k_groups<<<(unsigned)B, 1024, smem, s>>>(v, perm, (int)N, (int)K, gs);
  return last_launch_status();
}

// K8: prototype of each group (Eq. lite_select):
//   s_q = argmin_{t in G_q} sum_{j in G_q} v_j C(t, j), lowest index on ties,
// with C exactly as in the cost kernels.
//
// Scores of the members a = w, w + nwarps, ... of a group (warp w), each a
// full-width dot product per pair; the sum over targets runs in group
// order.  Keeps the warp's best (score, token).
template <typename T>
__device__ __forceinline__ void lite_proto_simt(const T* F, const float* inv, const float* X,
                                                const int32_t* TAU, const float* v,
                                                const int32_t* mem, int sz, const SceneNorms& nm,
                                                const DevParams& P, int D, int w, int lane,
                                                int nwarps, float& best, int& best_t) {
  constexpr int V = Vec16<T>::n;
  for (int a = w; a < sz; a += nwarps) {
    const int t = mem[a];
    const T* ft = F + (size_t)t * D;
    const float xt = X[3 * t], yt = X[3 * t + 1], zt = X[3 * t + 2];
    const int tt = TAU[t];
    const float inv_t = inv[t];
    float sc = 0.0f;
    for (int c = 0; c < sz; ++c) {
      const int j = mem[c];
      const T* fj = F + (size_t)j * D;
      float dot = 0.0f;
      for (int d = lane * V; d < D; d += 32 * V) {
        float x[V], y[V];
        Vec16<T>::load(ft + d, x);
        Vec16<T>::load(fj + d, y);
#pragma unroll
        for (int i = 0; i < V; ++i) dot = fmaf(x[i], y[i], dot);
      }
      dot = warp_sum(dot);
      float cosv = clamp_cos(dot * inv_t * inv[j]);
      if (t == j && inv_t > 0.0f) cosv = 1.0f;
      const float d2 = sqdist_rn(xt, yt, zt, X[3 * j], X[3 * j + 1], X[3 * j + 2]);
      sc += v[j] * fst_cost_from(cosv, d2, tt, TAU[j], nm, P);
    }
    if (sc < best || (sc == best && t < best_t)) {
      best = sc;
      best_t = t;
    }
  }
}

// One block per group, one warp per candidate (fp32 features, and bf16
// groups of more than LP_MAXG members).
template <typename T>
__global__ void __launch_bounds__(256) k_lite_proto(
    const T* __restrict__ F_all, const float* __restrict__ inv_all, const float* __restrict__ pos_all,
    const int32_t* __restrict__ frame_all, const SceneNorms* __restrict__ norms,
    const float* __restrict__ v_all, const int32_t* __restrict__ perm_all,
    const int32_t* __restrict__ gs_all, DevParams P, int N, int D, int K,
    int32_t* __restrict__ proto, double* __restrict__ score) {
  const int q = blockIdx.x, b = blockIdx.y;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int32_t* gs = gs_all + (size_t)b * (K + 1);
  const int sz = gs[q + 1] - gs[q];
  float best = INFINITY;
  int best_t = INT32_MAX;
  lite_proto_simt<T>(F_all + (size_t)b * N * D, inv_all + (size_t)b * N,
                     pos_all + (size_t)b * N * 3, frame_all + (size_t)b * N,
                     v_all + (size_t)b * N, perm_all + (size_t)b * N + gs[q], sz, norms[b], P, D,
                     w, lane, 8, best, best_t);
  __shared__ float s_sc[8];
  __shared__ int s_t[8];
  if (lane == 0) {
    s_sc[w] = best;
    s_t[w] = best_t;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < 8; ++i)
      if (s_sc[i] < best || (s_sc[i] == best && s_t[i] < best_t)) {
        best = s_sc[i];
        best_t = s_t[i];
      }
    proto[(size_t)b * K + q] = best_t;
    score[(size_t)b * K + q] = (double)best;
  }
}

// bf16 features: the group's feature Gram on the tensor cores (mma.sync
// m16n8k16, fp32 accumulate).  Members are taken in 16-row blocks and the
// 16 x 16 tiles (bi <= bj) of X X^T are computed one after the other, the
// feature width split over the block's 4 warps (warp w takes the 32-column
// chunks w, w + 4, ...) and the four partial tiles added in warp order.  In
// a chunk each lane loads 16 bytes of each of its rows (columns 8 (lane %
// 4) ..): those 8 values feed two k16 steps, the columns' order along k
// being the same for A and for B, so the dot products are unchanged.  A
// block against itself reuses its A registers as B.  The tiles land, both
// ways for bi < bj, in a shared-memory Gram, from which the scores read
// every pair's dot product once.  Groups of more than LP_MAXG members
// (rare: capacity-balanced groups are small) take the full-width loop.
constexpr int LP_MAXG = 64, LP_WARPS = 4;
__device__ __forceinline__ uint4 ld_row16(const __nv_bfloat16* row, int col, int D) {
  return (row != nullptr && col < D) ? __ldg(reinterpret_cast<const uint4*>(row + col))
                                     : make_uint4(0u, 0u, 0u, 0u);
}
// ld_row16 as an asynchronous copy into shared memory (zeros where it gives
// zeros: no bytes are read then, and F itself stands in as the source)
__device__ __forceinline__ void cp_row16(uint4* dst, const __nv_bfloat16* row, int col, int D,
                                         const void* any) {
  const bool ok = row != nullptr && col < D;
  cp_async16_zfill(dst, ok ? (const void*)(row + col) : any, ok);
}
constexpr int LP_STAGES = 4;  // chunks of a warp in flight (diagonal tiles)
__global__ void __launch_bounds__(32 * LP_WARPS) k_lite_proto_tc(
    const __nv_bfloat16* __restrict__ F_all, const float* __restrict__ inv_all,
    const float* __restrict__ pos_all, const int32_t* __restrict__ frame_all,
    const SceneNorms* __restrict__ norms, const float* __restrict__ v_all,
    const int32_t* __restrict__ perm_all, const int32_t* __restrict__ gs_all, DevParams P, int N,
    int D, int K, int32_t* __restrict__ proto, double* __restrict__ score) {
  __shared__ float s_dot[LP_MAXG][LP_MAXG + 1];
  __shared__ float s_part[LP_WARPS][16][17];
  // diagonal tiles: each lane's two 16-byte pieces of a chunk, LP_STAGES deep
  __shared__ __align__(16) uint4 s_stg[LP_WARPS][LP_STAGES][2][32];
  __shared__ float s_inv[LP_MAXG], s_v[LP_MAXG], s_x[LP_MAXG][3];
  __shared__ int s_mem[LP_MAXG], s_tau[LP_MAXG];
  __shared__ float s_sc[LP_WARPS];
  __shared__ int s_t[LP_WARPS];
  const int q = blockIdx.x, b = blockIdx.y;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const __nv_bfloat16* F = F_all + (size_t)b * N * D;
  const float* inv = inv_all + (size_t)b * N;
  const float* X = pos_all + (size_t)b * N * 3;
  const int32_t* TAU = frame_all + (size_t)b * N;
  const float* v = v_all + (size_t)b * N;
  const int32_t* gs = gs_all + (size_t)b * (K + 1);
  const int32_t* mem = perm_all + (size_t)b * N + gs[q];
  const int sz = gs[q + 1] - gs[q];
  const SceneNorms nm = norms[b];
  float best = INFINITY;
  int best_t = INT32_MAX;
  if (sz > LP_MAXG) {
    lite_proto_simt<__nv_bfloat16>(F, inv, X, TAU, v, mem, sz, nm, P, D, w, lane, LP_WARPS, best,
                                   best_t);
  } else {
    for (int a = threadIdx.x; a < sz; a += blockDim.x) {
      const int t = mem[a];
      s_mem[a] = t;
      s_inv[a] = inv[t];
      s_v[a] = v[t];
      s_x[a][0] = X[3 * t];
      s_x[a][1] = X[3 * t + 1];
      s_x[a][2] = X[3 * t + 2];
      s_tau[a] = TAU[t];
    }
    __syncthreads();
    const int g = lane >> 2, tg = lane & 3;
    const int nb = (sz + 15) >> 4;
    for (int bi = 0; bi < nb; ++bi) {
      for (int bj = bi; bj < nb; ++bj) {
        const int ra0 = 16 * bi + g, ra1 = ra0 + 8, rb0 = 16 * bj + g, rb1 = rb0 + 8;
        const __nv_bfloat16* pa0 = ra0 < sz ? F + (size_t)s_mem[ra0] * D : nullptr;
        const __nv_bfloat16* pa1 = ra1 < sz ? F + (size_t)s_mem[ra1] * D : nullptr;
        const __nv_bfloat16* pb0 = rb0 < sz ? F + (size_t)s_mem[rb0] * D : nullptr;
        const __nv_bfloat16* pb1 = rb1 < sz ? F + (size_t)s_mem[rb1] * D : nullptr;
        float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f};
        if (bi == bj) {
          // diagonal tile (B rows are A's): the same chunks and MMAs as the
          // loop below, the rows brought in by asynchronous copies
          // LP_STAGES chunks ahead (each lane reads back only its own copies)
          const int nch = (D - 32 * w + 32 * LP_WARPS - 1) / (32 * LP_WARPS);
          auto issue = [&](int i) {
            const int col = 32 * w + 32 * LP_WARPS * i + 8 * tg;
            cp_row16(&s_stg[w][i % LP_STAGES][0][lane], pa0, col, D, F);
            cp_row16(&s_stg[w][i % LP_STAGES][1][lane], pa1, col, D, F);
          };
#pragma unroll
          for (int i = 0; i < LP_STAGES - 1; ++i) {
            if (i < nch) issue(i);
            cp_commit();
          }
          for (int i = 0; i < nch; ++i) {
            if (i + LP_STAGES - 1 < nch) issue(i + LP_STAGES - 1);
            cp_commit();
            cp_wait<LP_STAGES - 1>();  // chunk i has landed
            const uint4 x0 = s_stg[w][i % LP_STAGES][0][lane];
            const uint4 x1 = s_stg[w][i % LP_STAGES][1][lane];
            mma_bf16_16816(d0, x0.x, x1.x, x0.y, x1.y, x0.x, x0.y);
            mma_bf16_16816(d1, x0.x, x1.x, x0.y, x1.y, x1.x, x1.y);
            mma_bf16_16816(d0, x0.z, x1.z, x0.w, x1.w, x0.z, x0.w);
            mma_bf16_16816(d1, x0.z, x1.z, x0.w, x1.w, x1.z, x1.w);
          }
          cp_wait<0>();
        }
        // off-diagonal tiles (groups of more than 16): A and B rows loaded
#pragma unroll 2
        for (int c0 = 32 * w; bi != bj && c0 < D; c0 += 32 * LP_WARPS) {
          const int col = c0 + 8 * tg;
          const uint4 x0 = ld_row16(pa0, col, D), x1 = ld_row16(pa1, col, D);
          const uint4 y0 = ld_row16(pb0, col, D), y1 = ld_row16(pb1, col, D);
          // k16 step over columns 8 tg + {0..3} of every lane, then + {4..7}
          mma_bf16_16816(d0, x0.x, x1.x, x0.y, x1.y, y0.x, y0.y);
          mma_bf16_16816(d1, x0.x, x1.x, x0.y, x1.y, y1.x, y1.y);
          mma_bf16_16816(d0, x0.z, x1.z, x0.w, x1.w, y0.z, y0.w);
          mma_bf16_16816(d1, x0.z, x1.z, x0.w, x1.w, y1.z, y1.w);
        }
        // d0: tile rows g (d0[0..1]) and g + 8 (d0[2..3]), columns 2 tg + {0, 1};
        // d1: the same rows, columns 8 + 2 tg + {0, 1}
        s_part[w][g][2 * tg] = d0[0];
        s_part[w][g][2 * tg + 1] = d0[1];
        s_part[w][g + 8][2 * tg] = d0[2];
        s_part[w][g + 8][2 * tg + 1] = d0[3];
        s_part[w][g][8 + 2 * tg] = d1[0];
        s_part[w][g][9 + 2 * tg] = d1[1];
        s_part[w][g + 8][8 + 2 * tg] = d1[2];
        s_part[w][g + 8][9 + 2 * tg] = d1[3];
        __syncthreads();
        for (int e = threadIdx.x; e < 256; e += blockDim.x) {
          const int r = e >> 4, c = e & 15;
          const int rr = 16 * bi + r, cc = 16 * bj + c;
          if (rr < sz && cc < sz) {
            const float x = ((s_part[0][r][c] + s_part[1][r][c]) + s_part[2][r][c]) +
                            s_part[3][r][c];
            s_dot[rr][cc] = x;
            if (bi != bj) s_dot[cc][rr] = x;
          }
        }
        __syncthreads();  // s_part is reused by the next tile
      }
    }
    for (int a = w; a < sz; a += LP_WARPS) {
      const int t = s_mem[a];
      const float inv_t = s_inv[a];
      float sc = 0.0f;
      for (int c = lane; c < sz; c += 32) {
        float cosv = clamp_cos(s_dot[a][c] * inv_t * s_inv[c]);
        if (c == a && inv_t > 0.0f) cosv = 1.0f;
        const float d2 = sqdist_rn(s_x[a][0], s_x[a][1], s_x[a][2], s_x[c][0], s_x[c][1],
                                   s_x[c][2]);
        sc += s_v[c] * fst_cost_from(cosv, d2, s_tau[a], s_tau[c], nm, P);
      }
      sc = warp_sum(sc);
      if (sc < best || (sc == best && t < best_t)) {
        best = sc;
        best_t = t;
      }
    }
  }
  if (lane == 0) {
    s_sc[w] = best;
    s_t[w] = best_t;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < LP_WARPS; ++i)
      if (s_sc[i] < best || (s_sc[i] == best && s_t[i] < best_t)) {
        best = s_sc[i];
        best_t = s_t[i];
      }
    proto[(size_t)b * K + q] = best_t;
    score[(size_t)b * K + q] = (double)best;
  }
}

// Lite objective: sum of the group scores, fp64, fixed order.
__global__ void __launch_bounds__(256) k_sum_scores(const double* __restrict__ score, int K,
                                                    double* __restrict__ objective) {
  const int b = blockIdx.x;
  double acc = 0.0;
  for (int q = threadIdx.x; q < K; q += blockDim.x) acc += score[(size_t)b * K + q];
  acc = warp_sum(acc);
  __shared__ double s[8];
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < 8; ++i) t += s[i];
    objective[b] = t;
  }
}

int launch_lite_proto(const void* feats, int dtype, const float* inv, const float* pos,
                      const int32_t* frame, const SceneNorms* norms, const float* v,
                      const int32_t* perm, const int32_t* gs, const DevParams& P, int64_t B,
                      int64_t N, int64_t D, int64_t K, int32_t* proto, double* score,
                      double* objective, cudaStream_t s) {
  dim3 grid((unsigned)K, (unsigned)B);
  if (dtype == CP_BF16)
    k_lite_proto_tc<<<grid, 32 * LP_WARPS, 0, s>>>((const __nv_bfloat16*)feats, inv, pos, frame,
                                                   norms, v, perm, gs, P, (int)N, (int)D, (int)K,
                                                   proto, score);
  else
    k_lite_proto<float><<<grid, 256, 0, s>>>((const float*)feats, inv, pos, frame, norms, v, perm,
                                             gs, P, (int)N, (int)D, (int)K, proto, score);
  int st = last_launch_status();
  if (st != CP_OK || !objective) return st;
  k_sum_scores<<<(unsigned)B, 256, 0, s>>>(score, (int)K, objective);
  return last_launch_status();
}

}  // namespace cp
