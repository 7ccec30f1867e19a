// K0 (scene statistics, inverse feature norms), K1 (3D nearest neighbours and
// scene diameter) and the min-max normalisers of Sec. 3.3.
#include "common.cuh"
#include "bf16_dot.cuh"

namespace cp {

// ---------------------------------------------------------------------------
// K0a: frame range (0 when frame is NULL) and bounding-box minimum per scene;
// initialises the fields that later kernels reduce into atomically.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(512) k_scene_stats(const float* __restrict__ pos,
                                                     const int32_t* __restrict__ frame,
                                                     int N, SceneStats* stats) {
  const int b = blockIdx.x;
  const float* X = pos + (size_t)b * N * 3;
  const int32_t* T = frame ? frame + (size_t)b * N : nullptr;  // may be absent
  int tmin = INT32_MAX, tmax = INT32_MIN;
  float lo[3] = {INFINITY, INFINITY, INFINITY};
  for (int j0 = threadIdx.x; j0 < N; j0 += 4 * 512) {  // four tokens' loads in flight
    int t[4];
    float x[4][3];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = min(j0 + 512 * u, N - 1);
      t[u] = T ? T[j] : 0;
#pragma unroll
      for (int a = 0; a < 3; ++a) x[u][a] = X[3 * j + a];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      tmin = min(tmin, t[u]);
      tmax = max(tmax, t[u]);
#pragma unroll
      for (int a = 0; a < 3; ++a) lo[a] = fminf(lo[a], x[u][a]);
    }
  }
  __shared__ int s_tmin[16], s_tmax[16];
  __shared__ float s_lo[3][16];
  for (int o = 16; o > 0; o >>= 1) {
    tmin = min(tmin, __shfl_xor_sync(0xFFFFFFFFu, tmin, o));
    tmax = max(tmax, __shfl_xor_sync(0xFFFFFFFFu, tmax, o));
#pragma unroll
    for (int a = 0; a < 3; ++a) lo[a] = fminf(lo[a], __shfl_xor_sync(0xFFFFFFFFu, lo[a], o));
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) {
    s_tmin[w] = tmin;
    s_tmax[w] = tmax;
    for (int a = 0; a < 3; ++a) s_lo[a][w] = lo[a];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const int nw = blockDim.x >> 5;
    for (int i = 1; i < nw; ++i) {
      tmin = min(tmin, s_tmin[i]);
      tmax = max(tmax, s_tmax[i]);
      for (int a = 0; a < 3; ++a) lo[a] = fminf(lo[a], s_lo[a][i]);
    }
    SceneStats st;
    st.cos_max_key = 0u;           // below every real key
    st.cos_min_key = 0xFFFFFFFFu;  // above every real key
    st.d2_max_bits = 0u;           // d^2 >= 0: float bits order like the values
    st.tau_min = tmin;
    st.tau_max = tmax;
    for (int a = 0; a < 3; ++a) st.bbox_min[a] = lo[a];
    for (int i = 0; i < 8; ++i) st.pad[i] = 0u;
    stats[b] = st;
  }
}

int launch_scene_stats(const float* pos, const int32_t* frame, int64_t B, int64_t N,
                       SceneStats* stats, cudaStream_t s) {
  k_scene_stats<<<(unsigned)B, 512, 0, s>>>(pos, frame, (int)N, stats);
  return last_launch_status();
}

// ---------------------------------------------------------------------------
// K0b: inv[j] = 1 / ||f_j|| (0 for a zero feature), one warp per token.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) k_inv_norms(const T* __restrict__ F,
                                                   const float* __restrict__ pos, int64_t rows,
                                                   int D, float* __restrict__ inv,
                                                   float4* __restrict__ tok) {
  const int64_t row = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= rows) return;
  const T* f = F + row * D;
  constexpr int V = Vec16<T>::n;
  float acc = 0.0f;
  if constexpr (V == 8) {  // bf16: the same products and order, no widening
    for (int d = lane * V; d < D; d += 32 * V) {
      const uint4 x = __ldg(reinterpret_cast<const uint4*>(f + d));
      acc = dot8_bf16(x, x, acc);
    }
  } else {
    for (int d = lane * V; d < D; d += 32 * V) {
      float x[V];
      Vec16<T>::load(f + d, x);
#pragma unroll
      for (int i = 0; i < V; ++i) acc = fmaf(x[i], x[i], acc);
    }
  }
  acc = warp_sum(acc);
  if (lane == 0) {
    const float iv = acc > 0.0f ? 1.0f / sqrtf(acc) : 0.0f;
    inv[row] = iv;
    if (tok) tok[row] = make_float4(pos[3 * row], pos[3 * row + 1], pos[3 * row + 2], iv);
  }
}

int launch_inv_norms(const void* feats, int dtype, const float* pos, int64_t B, int64_t N,
                     int64_t D, float* inv, float4* tok, cudaStream_t s) {
  const int64_t rows = B * N;
  const unsigned grid = (unsigned)((rows + 7) / 8);
  if (dtype == CP_BF16)
    k_inv_norms<__nv_bfloat16><<<grid, 256, 0, s>>>((const __nv_bfloat16*)feats, pos, rows,
                                                     (int)D, inv, tok);
  else
    k_inv_norms<float><<<grid, 256, 0, s>>>((const float*)feats, pos, rows, (int)D, inv, tok);
  return last_launch_status();
}

// ---------------------------------------------------------------------------
// K1: for token j, its kk nearest other tokens ordered by (fp32 d^2, index)
// (capacity set N_n of Eq. fst_capacity_score and SGS neighbourhood M_g of
// Eq. local_neighbor), and the largest squared distance of the row (for the
// spatial normaliser).  One block per token; the N keys live in shared
// memory; the kk-th smallest key is found by bisection on its bit pattern
// (d^2 >= 0, so float bits order like the values), the winners are collected
// in index order and sorted by (key, index).
// ---------------------------------------------------------------------------
constexpr int KNN_THREADS = 256;

__device__ __forceinline__ int block_sum_int(int v, int* s_red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) s_red[w] = v;
  __syncthreads();
  int t = 0;
  for (int i = 0; i < KNN_THREADS / 32; ++i) t += s_red[i];
  return t;
}

__global__ void __launch_bounds__(KNN_THREADS) k_knn(const float* __restrict__ pos, int N, int kk,
                                                     int list_len, int32_t* __restrict__ nbr,
                                                     SceneStats* stats) {
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned long long* list = reinterpret_cast<unsigned long long*>(smem);  // [list_len]
  uint32_t* key = reinterpret_cast<uint32_t*>(list + list_len);            // [N]
  __shared__ int s_red[KNN_THREADS / 32];
  __shared__ uint32_t s_redu[KNN_THREADS / 32];
  __shared__ int s_wcnt[2][KNN_THREADS / 32];

  const int j = blockIdx.x, b = blockIdx.y;
  const float* X = pos + (size_t)b * N * 3;
  const float xj = X[3 * j], yj = X[3 * j + 1], zj = X[3 * j + 2];
  uint32_t dmax = 0u;
  for (int k = threadIdx.x; k < N; k += KNN_THREADS) {
    float d2 = sqdist_rn(xj, yj, zj, X[3 * k], X[3 * k + 1], X[3 * k + 2]);
    uint32_t bits = __float_as_uint(d2);
    dmax = max(dmax, bits);
    key[k] = (k == j) ? 0xFFFFFFFFu : bits;
  }
  for (int o = 16; o > 0; o >>= 1) dmax = max(dmax, __shfl_xor_sync(0xFFFFFFFFu, dmax, o));
  if ((threadIdx.x & 31) == 0) s_redu[threadIdx.x >> 5] = dmax;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < KNN_THREADS / 32; ++i) dmax = max(dmax, s_redu[i]);
    atomicMax(&stats[b].d2_max_bits, dmax);
  }
  if (kk <= 0) return;

  // bisection: smallest T with #{key <= T} >= kk
  uint32_t lo = 0u, hi = 0xFFFFFFFEu;
  while (lo < hi) {
    const uint32_t mid = lo + ((hi - lo) >> 1);
    int c = 0;
    for (int k = threadIdx.x; k < N; k += KNN_THREADS) c += key[k] <= mid;
    c = block_sum_int(c, s_red);
    if (c >= kk) hi = mid; else lo = mid + 1;
  }
  const uint32_t T = lo;
  int less = 0;
  for (int k = threadIdx.x; k < N; k += KNN_THREADS) less += key[k] < T;
  less = block_sum_int(less, s_red);
  const int need_eq = kk - less;

  // collect in index order: every key < T, and the first need_eq keys == T
  for (int i = threadIdx.x; i < list_len; i += KNN_THREADS) list[i] = ~0ull;
  __syncthreads();
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  int base = 0, eq_taken = 0;
  for (int c0 = 0; c0 < N; c0 += KNN_THREADS) {
    const int k = c0 + threadIdx.x;
    const uint32_t kv = k < N ? key[k] : 0xFFFFFFFFu;
    const bool is_eq = kv == T && k < N;
    // rank among equal keys of this chunk, in index order
    const unsigned beq = __ballot_sync(0xFFFFFFFFu, is_eq);
    if (l == 0) s_wcnt[0][w] = __popc(beq);
    __syncthreads();
    int eq_before = 0, eq_total = 0;
    for (int i = 0; i < KNN_THREADS / 32; ++i) {
      eq_before += i < w ? s_wcnt[0][i] : 0;
      eq_total += s_wcnt[0][i];
    }
    const int rank_eq = eq_taken + eq_before + __popc(beq & ((1u << l) - 1u));
    const bool take = (kv < T && k < N) || (is_eq && rank_eq < need_eq);
    const unsigned bt = __ballot_sync(0xFFFFFFFFu, take);
    if (l == 0) s_wcnt[1][w] = __popc(bt);
    __syncthreads();
    int t_before = 0, t_total = 0;
    for (int i = 0; i < KNN_THREADS / 32; ++i) {
      t_before += i < w ? s_wcnt[1][i] : 0;
      t_total += s_wcnt[1][i];
    }
    if (take) {
      const int p = base + t_before + __popc(bt & ((1u << l) - 1u));
      list[p] = ((unsigned long long)kv << 32) | (unsigned)k;
    }
    base += t_total;
    eq_taken += eq_total;
    __syncthreads();
  }
  // bitonic sort of list[0, list_len) ascending by (key, index)
  for (int size = 2; size <= list_len; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int i = threadIdx.x; i < (list_len >> 1); i += KNN_THREADS) {
        const int a = 2 * i - (i & (stride - 1));
        const int c = a + stride;
        const bool up = (a & size) == 0;
        const unsigned long long x = list[a], y = list[c];
        if ((x > y) == up) { list[a] = y; list[c] = x; }
      }
      __syncthreads();
    }
  }
  int32_t* out = nbr + ((size_t)b * N + j) * kk;
  for (int q = threadIdx.x; q < kk; q += KNN_THREADS) out[q] = (int32_t)(list[q] & 0xFFFFFFFFu);
}

// K1 for kk <= 32: one warp per token.  Each lane scans every 32nd candidate
// and keeps its KK smallest (d^2 bits, index) keys in registers, sorted; the
// warp then merges the 32 lists by repeated warp-wide minimum.  The keys are
// the same total order as the block kernel's, so the lists are identical.
template <int KK>
__global__ void __launch_bounds__(256) k_knn_warp(const float* __restrict__ pos, int N, int kk,
                                                  int32_t* __restrict__ nbr, SceneStats* stats) {
  const int j = blockIdx.x * 8 + (threadIdx.x >> 5);
  const int b = blockIdx.y;
  const int lane = threadIdx.x & 31;
  const float* X = pos + (size_t)b * N * 3;
  uint32_t dmax = 0u;
  if (j < N) {
    const float xj = X[3 * j], yj = X[3 * j + 1], zj = X[3 * j + 2];
    unsigned long long best[KK];
#pragma unroll
    for (int i = 0; i < KK; ++i) best[i] = ~0ull;
    for (int k = lane; k < N; k += 32) {
      const float d2 = sqdist_rn(xj, yj, zj, __ldg(X + 3 * k), __ldg(X + 3 * k + 1),
                                 __ldg(X + 3 * k + 2));
      const uint32_t bits = __float_as_uint(d2);
      dmax = max(dmax, bits);
      const unsigned long long key = ((unsigned long long)bits << 32) | (uint32_t)k;
      if (k != j && key < best[KK - 1]) {
        best[KK - 1] = key;
#pragma unroll
        for (int i = KK - 1; i > 0; --i) {
          if (best[i] < best[i - 1]) {
            const unsigned long long t = best[i];
            best[i] = best[i - 1];
            best[i - 1] = t;
          }
        }
      }
    }
    int32_t* out = nbr + ((size_t)b * N + j) * kk;
    for (int q = 0; q < kk; ++q) {
      const unsigned long long m = warp_min_u64(best[0]);
      if (lane == 0) out[q] = (int32_t)(m & 0xFFFFFFFFull);
      if (best[0] == m) {  // keys are unique: exactly one lane pops its head
#pragma unroll
        for (int i = 0; i < KK - 1; ++i) best[i] = best[i + 1];
        best[KK - 1] = ~0ull;
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) dmax = max(dmax, __shfl_xor_sync(0xFFFFFFFFu, dmax, o));
  __shared__ uint32_t s_dmax[8];
  if (lane == 0) s_dmax[threadIdx.x >> 5] = dmax;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t m = s_dmax[0];
    for (int i = 1; i < 8; ++i) m = max(m, s_dmax[i]);
    atomicMax(&stats[b].d2_max_bits, m);
  }
}

// K1 for kk <= 8, two tokens per warp, 16 per block: the block stages the
// candidate positions in shared-memory tiles of 2048, so each position is
// read from L2 once per 16 query rows; the quick test on the d^2 bits skips
// the 64-bit key compare for almost every candidate.  Same keys, same lists
// as k_knn_warp.
constexpr int KNN_TILE = 2048;

template <int KK>
__global__ void __launch_bounds__(256) k_knn_pair(const float* __restrict__ pos, int N, int kk,
                                                  int32_t* __restrict__ nbr, SceneStats* stats) {
  __shared__ float4 s_p[KNN_TILE];
  const int j0 = (blockIdx.x * 8 + (threadIdx.x >> 5)) * 2;
  const int b = blockIdx.y;
  const int lane = threadIdx.x & 31;
  const float* X = pos + (size_t)b * N * 3;
  const bool active = j0 < N;
  const bool two = j0 + 1 < N;
  const int j1 = two ? j0 + 1 : j0;
  float ax = 0.f, ay = 0.f, az = 0.f, bx = 0.f, by = 0.f, bz = 0.f;
  if (active) {
    ax = X[3 * j0]; ay = X[3 * j0 + 1]; az = X[3 * j0 + 2];
    bx = X[3 * j1]; by = X[3 * j1 + 1]; bz = X[3 * j1 + 2];
  }
  uint32_t dmax = 0u;
  unsigned long long best0[KK], best1[KK];
#pragma unroll
  for (int i = 0; i < KK; ++i) best0[i] = best1[i] = ~0ull;
  for (int base = 0; base < N; base += KNN_TILE) {
    const int n = min(KNN_TILE, N - base);
    __syncthreads();  // the previous tile is consumed
    for (int i = threadIdx.x; i < n; i += 256) {
      const int k = base + i;
      s_p[i] = make_float4(__ldg(X + 3 * k), __ldg(X + 3 * k + 1), __ldg(X + 3 * k + 2), 0.f);
    }
    __syncthreads();
    if (!active) continue;
    for (int i = lane; i < n; i += 32) {
      const int k = base + i;
      const float4 p = s_p[i];
      const uint32_t ba = __float_as_uint(sqdist_rn(ax, ay, az, p.x, p.y, p.z));
      const uint32_t bb = __float_as_uint(sqdist_rn(bx, by, bz, p.x, p.y, p.z));
      dmax = max(dmax, max(ba, bb));
      if (ba <= (uint32_t)(best0[KK - 1] >> 32) && k != j0) {
        const unsigned long long key = ((unsigned long long)ba << 32) | (uint32_t)k;
        if (key < best0[KK - 1]) {
          best0[KK - 1] = key;
#pragma unroll
          for (int t = KK - 1; t > 0; --t)
            if (best0[t] < best0[t - 1]) {
              const unsigned long long x = best0[t];
              best0[t] = best0[t - 1];
              best0[t - 1] = x;
            }
        }
      }
      if (bb <= (uint32_t)(best1[KK - 1] >> 32) && k != j1) {
        const unsigned long long key = ((unsigned long long)bb << 32) | (uint32_t)k;
        if (key < best1[KK - 1]) {
          best1[KK - 1] = key;
#pragma unroll
          for (int t = KK - 1; t > 0; --t)
            if (best1[t] < best1[t - 1]) {
              const unsigned long long x = best1[t];
              best1[t] = best1[t - 1];
              best1[t - 1] = x;
            }
        }
      }
    }
  }
  if (active && nbr) {
    int32_t* out0 = nbr + ((size_t)b * N + j0) * kk;
    for (int q = 0; q < kk; ++q) {
      const unsigned long long m = warp_min_u64(best0[0]);
      if (lane == 0) out0[q] = (int32_t)(m & 0xFFFFFFFFull);
      if (best0[0] == m) {  // keys are unique: exactly one lane pops its head
#pragma unroll
        for (int i = 0; i < KK - 1; ++i) best0[i] = best0[i + 1];
        best0[KK - 1] = ~0ull;
      }
    }
    if (two) {
      int32_t* out1 = nbr + ((size_t)b * N + j1) * kk;
      for (int q = 0; q < kk; ++q) {
        const unsigned long long m = warp_min_u64(best1[0]);
        if (lane == 0) out1[q] = (int32_t)(m & 0xFFFFFFFFull);
        if (best1[0] == m) {
#pragma unroll
          for (int i = 0; i < KK - 1; ++i) best1[i] = best1[i + 1];
          best1[KK - 1] = ~0ull;
        }
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) dmax = max(dmax, __shfl_xor_sync(0xFFFFFFFFu, dmax, o));
  __shared__ uint32_t s_dmax[8];
  if (lane == 0) s_dmax[threadIdx.x >> 5] = dmax;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t m = s_dmax[0];
    for (int i = 1; i < 8; ++i) m = max(m, s_dmax[i]);
    atomicMax(&stats[b].d2_max_bits, m);
  }
}

int launch_knn(const float* pos, int64_t B, int64_t N, int kk, int32_t* nbr, SceneStats* stats,
               cudaStream_t s) {
  if (kk <= 8) {
    dim3 grid((unsigned)((N + 15) / 16), (unsigned)B);
    k_knn_pair<8><<<grid, 256, 0, s>>>(pos, (int)N, kk, nbr, stats);
    return last_launch_status();
  }
  if (kk <= 32) {
    dim3 grid((unsigned)((N + 7) / 8), (unsigned)B);
    if (kk <= 16)
      k_knn_warp<16><<<grid, 256, 0, s>>>(pos, (int)N, kk, nbr, stats);
    else
      k_knn_warp<32><<<grid, 256, 0, s>>>(pos, (int)N, kk, nbr, stats);
    return last_launch_status();
  }
  int list_len = 1;
  while (list_len < kk) list_len <<= 1;
  if (list_len < 2) list_len = 2;
  const size_t smem = sizeof(unsigned long long) * list_len + sizeof(uint32_t) * (size_t)N;
  CP_TRY_STATUS(allow_smem((const void*)k_knn, smem, "launch_knn: smem attribute"));
  dim3 grid((unsigned)N, (unsigned)B);
  k_knn<<<grid, KNN_THREADS, smem, s>>>(pos, (int)N, kk, list_len, nbr, stats);
  return last_launch_status();
}

// ---------------------------------------------------------------------------
// K1 through a uniform grid (kk <= kKnnGridMax): exact, with the same keys and lists
// as the brute-force kernels, but each query visits only the cells around
// it.  The scene's bounding box is cut into cubic cells of side h =
// (largest extent) / G with G = the least integer such that 4 G^3 >= N, so
// at most G^3 cells; points are counting-sorted by cell.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int grid_side(int N) {
  int G = 1;
  while (4 * G * G * G < N) ++G;
  return G;
}

// One block per scene: bounding box, cell size, counting sort by cell.  Bound
// by latency: three passes over the points, four points' loads in flight a
// thread, and a scan of the cell counts by all threads (one thread's scan
// was half of the time): 16384 points 21 us, 34 before; 1024 points 8 us.
__global__ void __launch_bounds__(1024) k_grid_build(const float* __restrict__ pos, int N,
                                                     int gmax, GridInfo* __restrict__ info,
                                                     int32_t* __restrict__ cell_start,
                                                     float4* __restrict__ sorted) {
  extern __shared__ int s_cnt[];  // [gmax + 1]
  __shared__ float s_red[6][32];
  const int b = blockIdx.x;
  const float* X = pos + (size_t)b * N * 3;
  float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  for (int j0 = threadIdx.x; j0 < N; j0 += 4 * 1024) {
    float x[4][3];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = min(j0 + 1024 * u, N - 1);
#pragma unroll
      for (int a = 0; a < 3; ++a) x[u][a] = X[3 * j + a];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        lo[a] = fminf(lo[a], x[u][a]);
        hi[a] = fmaxf(hi[a], x[u][a]);
      }
  }
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      lo[a] = fminf(lo[a], __shfl_xor_sync(0xFFFFFFFFu, lo[a], o));
      hi[a] = fmaxf(hi[a], __shfl_xor_sync(0xFFFFFFFFu, hi[a], o));
    }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0)
    for (int a = 0; a < 3; ++a) {
      s_red[a][w] = lo[a];
      s_red[3 + a][w] = hi[a];
    }
  for (int c = threadIdx.x; c <= gmax; c += blockDim.x) s_cnt[c] = 0;
  __syncthreads();
  __shared__ GridInfo s_g;
  if (threadIdx.x == 0) {
    const int nw = blockDim.x >> 5;
    for (int i = 1; i < nw; ++i)
      for (int a = 0; a < 3; ++a) {
        s_red[a][0] = fminf(s_red[a][0], s_red[a][i]);
        s_red[3 + a][0] = fmaxf(s_red[3 + a][0], s_red[3 + a][i]);
      }
    const int G = grid_side(N);
    float ext = 0.0f;
    for (int a = 0; a < 3; ++a) ext = fmaxf(ext, s_red[3 + a][0] - s_red[a][0]);
    GridInfo g;
    g.h = ext > 0.0f ? ext / (float)G : 1.0f;
    g.inv_h = 1.0f / g.h;
    int nc = 1;
    for (int a = 0; a < 3; ++a) {
      g.lo[a] = s_red[a][0];
      const float e = s_red[3 + a][0] - s_red[a][0];
      int d = (int)ceilf(e * g.inv_h);
      d = d < 1 ? 1 : (d > G ? G : d);
      g.dims[a] = d;
      nc *= d;
    }
    g.ncells = nc;
    s_g = g;
    info[b] = g;
  }
  __syncthreads();
  const GridInfo g = s_g;
  for (int j0 = threadIdx.x; j0 < N; j0 += 4 * 1024) {
    float x[4][3];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = min(j0 + 1024 * u, N - 1);
#pragma unroll
      for (int a = 0; a < 3; ++a) x[u][a] = X[3 * j + a];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (j0 + 1024 * u < N) atomicAdd(&s_cnt[grid_cell(g, x[u])], 1);
  }
  __syncthreads();
  // exclusive scan of the counts, a run of cells a thread
  __shared__ int s_sum[32];
  {
    const int per = (g.ncells + 1023) >> 10;
    const int c0 = min(g.ncells, (int)threadIdx.x * per), c1 = min(g.ncells, c0 + per);
    int sum = 0;
    for (int c = c0; c < c1; ++c) sum += s_cnt[c];
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (l >= o) incl += t;
    }
    if (l == 31) s_sum[w] = incl;
    __syncthreads();
    int run = __reduce_add_sync(0xFFFFFFFFu, l < w ? s_sum[l] : 0) + incl - sum;
    for (int c = c0; c < c1; ++c) {
      const int n = s_cnt[c];
      s_cnt[c] = run;
      run += n;
    }
    if (threadIdx.x == 0) s_cnt[g.ncells] = N;
  }
  __syncthreads();
  int32_t* cs = cell_start + (size_t)b * (gmax + 1);
  for (int c = threadIdx.x; c <= g.ncells; c += blockDim.x) cs[c] = s_cnt[c];
  __syncthreads();
  float4* out = sorted + (size_t)b * N;
  for (int j0 = threadIdx.x; j0 < N; j0 += 4 * 1024) {
    float x[4][3];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = min(j0 + 1024 * u, N - 1);
#pragma unroll
      for (int a = 0; a < 3; ++a) x[u][a] = X[3 * j + a];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = j0 + 1024 * u;
      if (j < N)
        out[atomicAdd(&s_cnt[grid_cell(g, x[u])], 1)] =
            make_float4(x[u][0], x[u][1], x[u][2], __int_as_float(j));
    }
  }
}

// One warp per query token, queries in cell order.  Three scans of candidate
// ranges (a range is the cells of one (y, z) row, contiguous in the sorted
// points; the ranges of 32 rows are scanned as one flat sequence):
//  - the query's own cell if it has more than 2 kk points, else the smallest
//    block of 3, 5, ... cells a side around it with more than kk: a histogram
//    of the squared distances, 8 bins an octave, gives a bound U that at least
//    kk of them are below (16384 tokens, 8 neighbours: the whole preparation
//    124 us, 159 with blocks of 3 cells a side at least, 122 / 130 with the
//    own cell from kk / 4 kk points on; 64 neighbours of 32 scenes 1.16 ms,
//    1.16, 1.28 / 1.17);
//  - every cell within sqrt(U) (rows and ends of rows by their distance, with
//    a margin for the rounding of the cell coordinates): the keys below U are
//    gathered, kk and usually a few more;
//  - should more than KW_CAP be (coincident points, say), histograms over the
//    range of those keys lower U until they fit.
// The gathered keys are ranked by counting; the first kk go out in order.
// Keys are (d^2 bits, index), as in the brute-force kernels.  Bound by
// instruction issue (a point costs ~40 instructions a scan, of the warp), no
// longer by the chain of one thread's scan and list: 56,000 queries (8 scenes
// of 7000), kk = 63: 0.17 ms, a heap per thread took 0.62; 262,144 queries:
// 0.82 (1.66); one scene of 8192, kk = 8: 0.017 (0.087), of 16384 0.041
// (0.37).
constexpr int KW_WARPS = 8, KW_CAP = 256;

__global__ void __launch_bounds__(32 * KW_WARPS) k_knn_grid(
    int N, int kk, int gmax, const GridInfo* __restrict__ info,
    const int32_t* __restrict__ cell_start, const float4* __restrict__ sorted,
    int32_t* __restrict__ nbr) {
  __shared__ __align__(16) unsigned long long s_buf[KW_WARPS][KW_CAP];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, b = blockIdx.y;
  const int jj = blockIdx.x * KW_WARPS + w;
  if (jj >= N) return;
  unsigned long long* buf = s_buf[w];
  uint32_t* hist = reinterpret_cast<uint32_t*>(buf);  // [256]
  const GridInfo g = info[b];
  const int32_t* cs = cell_start + (size_t)b * (gmax + 1);
  const float4* P = sorted + (size_t)b * N;
  const float4 qp = P[jj];
  const int self = __float_as_int(qp.w);
  const int cx = grid_coord(g, qp.x, 0), cy = grid_coord(g, qp.y, 1), cz = grid_coord(g, qp.z, 2);
  float span = 0.0f;
#pragma unroll
  for (int a = 0; a < 3; ++a) span = fmaxf(span, fabsf(g.lo[a]) + (float)g.dims[a] * g.h);
  const float delta = 1e-3f * g.h + 1e-5f * span;

  // The window of the next scan: rows [y0, y1] x [z0, z1], cells [x0, x1] of
  // them; rad2 < infinity: only cells within that distance.
  int x0, x1, y0, y1, z0, z1;
  float rad2;
  auto block = [&](int r) {
    x0 = max(cx - r, 0);
    x1 = min(cx + r, g.dims[0] - 1);
    y0 = max(cy - r, 0);
    y1 = min(cy + r, g.dims[1] - 1);
    z0 = max(cz - r, 0);
    z1 = min(cz + r, g.dims[2] - 1);
    rad2 = INFINITY;
  };
  // distance from the query to the cells of coordinate c along one axis
  auto gap = [&](int a, float q, int cq, int c) -> float {
    const float edge = g.lo[a] + (float)(c < cq ? c + 1 : c) * g.h;
    return c == cq ? 0.0f : fmaxf((c < cq ? q - edge : edge - q) - delta, 0.0f);
  };
  // Row q of the window: its first point and number of points.
  auto row = [&](int q, int rows, int ny, int& start) -> int {
    start = 0;
    if (q >= rows) return 0;
    const int z = z0 + q / ny, y = y0 + q % ny;
    int xa = x0, xb = x1;
    if (rad2 < INFINITY) {
      const float gy = gap(1, qp.y, cy, y), gz = gap(2, qp.z, cz, z);
      const float left = rad2 - (gy * gy + gz * gz);
      if (left < 0.0f) return 0;
      const float half = sqrtf(left) + delta;
      xa = max(xa, grid_coord(g, qp.x - half, 0));
      xb = min(xb, grid_coord(g, qp.x + half, 0));
    }
    const int base = (z * g.dims[1] + y) * g.dims[0];
    start = cs[base + xa];
    return cs[base + xb + 1] - start;
  };
  // visit(in, key) with the whole warp for every 32 points of the window
  auto scan = [&](auto&& visit) {
    const int ny = y1 - y0 + 1, rows = ny * (z1 - z0 + 1);
    for (int q0 = 0; q0 < rows; q0 += 32) {
      int start;
      const int len = row(q0 + lane, rows, ny, start);
      int incl = len;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += t;
      }
      const int total = __shfl_sync(0xFFFFFFFFu, incl, 31), excl = incl - len;
      for (int c0 = 0; c0 < total; c0 += 32) {
        const int c = min(c0 + lane, total - 1);
        int r = 0;  // the row of the c-th point: the last that starts at or before c
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
          if (__shfl_sync(0xFFFFFFFFu, excl, r + o) <= c) r += o;
        const float4 p =
            P[__shfl_sync(0xFFFFFFFFu, start, r) + c - __shfl_sync(0xFFFFFFFFu, excl, r)];
        const int k = __float_as_int(p.w);
        const uint32_t bits = __float_as_uint(sqdist_rn(qp.x, qp.y, qp.z, p.x, p.y, p.z));
        visit(c0 + lane < total && k != self, ((unsigned long long)bits << 32) | (uint32_t)k);
      }
    }
  };
  // the bin of hist in which the count reaches `want`, and the count before it
  auto bin_of = [&](int want, int& before) -> int {
    __syncwarp();
    const uint4 h0 = reinterpret_cast<const uint4*>(hist)[2 * lane];
    const uint4 h1 = reinterpret_cast<const uint4*>(hist)[2 * lane + 1];
    const uint32_t h[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
    uint32_t sum = 0u;
#pragma unroll
    for (int i = 0; i < 8; ++i) sum += h[i];
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += t;
    }
    const int first = __ffs(__ballot_sync(0xFFFFFFFFu, incl >= (uint32_t)want)) - 1;
    int bin = 0;
    uint32_t run = incl - sum, below = run;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      run += h[i];
      if (run < (uint32_t)want) {
        bin = i + 1;
        below = run;
      }
    }
    before = (int)__shfl_sync(0xFFFFFFFFu, below, first);
    return 8 * first + __shfl_sync(0xFFFFFFFFu, bin, first);
  };
  auto clear = [&]() {
    reinterpret_cast<uint4*>(hist)[2 * lane] = make_uint4(0u, 0u, 0u, 0u);
    reinterpret_cast<uint4*>(hist)[2 * lane + 1] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
  };

  // ---- a block with more than kk points (the query among them)
  for (int r = 0;; ++r) {
    block(r);
    const int ny = y1 - y0 + 1, rows = ny * (z1 - z0 + 1);
    int n = 0;
    for (int q = lane; q < rows; q += 32) {
      int start;
      n += row(q, rows, ny, start);
    }
    n = __reduce_add_sync(0xFFFFFFFFu, n);
    if (n > (r == 0 ? 2 * kk : kk)) break;  // N > kk: the whole grid at the latest
  }
  const float far = 64.0f * g.h;
  const int off = (int)(__float_as_uint(far * far) >> 20) - 255;
  clear();
  scan([&](bool in, unsigned long long key) {
    const int bin = min(max((int)(key >> 52) - off, 0), 255);
    if (in) atomicAdd(hist + bin, 1u);
  });
  int below;
  const int top = bin_of(kk, below);
  // at least kk keys are below U
  unsigned long long U = top == 255 ? ~0ull : (unsigned long long)(top + 1 + off) << 52;
  // ---- the keys below U; `sure` of the kk are below L
  unsigned long long L = 0ull;
  int n = 0, sure = 0;
  for (;;) {
    const float d2 = __uint_as_float((uint32_t)(U >> 32));
    if (d2 < 1e30f) {
      const float rad = sqrtf(d2) * 1.000244140625f + delta;  // 1 + 2^-12
      x0 = 0;
      x1 = g.dims[0] - 1;
      y0 = grid_coord(g, qp.y - rad, 1);
      y1 = grid_coord(g, qp.y + rad, 1);
      z0 = grid_coord(g, qp.z - rad, 2);
      z1 = grid_coord(g, qp.z + rad, 2);
      rad2 = rad * rad;
    } else {  // infinite or not a number: everywhere
      block(max(g.dims[0], max(g.dims[1], g.dims[2])));
    }
    n = 0;
    unsigned long long lo = ~0ull, hi = 0ull;
    scan([&](bool in, unsigned long long key) {
      in = in && key < U;
      const uint32_t mask = __ballot_sync(0xFFFFFFFFu, in);
      if (in) {
        const int at = n + __popc(mask & ((1u << lane) - 1u));
        if (at < KW_CAP) buf[at] = key;
        if (key >= L) {
          lo = key < lo ? key : lo;
          hi = key > hi ? key : hi;
        }
      }
      n += __popc(mask);
    });
    if (n <= KW_CAP) break;
    // too many: a histogram of those from L on over their range [lo, hi];
    // the bin with the kk-th is at most a 128th of it, down to a single key
    lo = __shfl_sync(0xFFFFFFFFu, warp_min_u64(lo), 0);
    hi = __shfl_sync(0xFFFFFFFFu, warp_max_u64(hi), 0);
    const int shift = max(0, 56 - __clzll((long long)((hi - lo) | 1ull)));
    __syncwarp();
    clear();
    scan([&](bool in, unsigned long long key) {
      if (in && key >= lo && key <= hi) atomicAdd(hist + (int)((key - lo) >> shift), 1u);
    });
    const int bin = bin_of(kk - sure, below);
    sure += below;
    L = lo + ((unsigned long long)bin << shift);
    U = L + (1ull << shift);
  }
  __syncwarp();
  // ---- ranks
  int32_t* out = nbr + ((size_t)b * N + self) * kk;
  for (int i0 = 0; i0 < n; i0 += 64) {
    const unsigned long long ka = i0 + lane < n ? buf[i0 + lane] : ~0ull;
    const unsigned long long kb = i0 + 32 + lane < n ? buf[i0 + 32 + lane] : ~0ull;
    int ra = 0, rb = 0;
#pragma unroll 4
    for (int t = 0; t < n; ++t) {
      const unsigned long long o = buf[t];
      ra += o < ka ? 1 : 0;
      rb += o < kb ? 1 : 0;
    }
    if (i0 + lane < n && ra < kk) out[ra] = (int32_t)(uint32_t)ka;
    if (i0 + 32 + lane < n && rb < kk) out[rb] = (int32_t)(uint32_t)kb;
  }
}

// Few neighbours (kk <= 8) of very many queries: one thread per query token
// scans the shells of cells at Chebyshev distance r = 0, 1, 2, ... from its
// own cell; every point outside the first r shells is more than r h away
// along some axis, so once the kk-th best squared distance is below ((r -
// 1/1024) h)^2 (the margin covers the rounding of the cell coordinates) no
// later point can enter the list.  The KK best keys are kept unsorted with the
// position of the worst: a closer point overwrites the worst (a select per
// slot, so the list stays in registers) and the worst is found again; the
// list is sorted once at the end.  Keys are (d^2 bits, index), as in the
// brute-force kernels.
template <int KK>
__global__ void __launch_bounds__(128) k_knn_grid_thread(int N, int kk, int gmax, const GridInfo* __restrict__ info,
                                                  const int32_t* __restrict__ cell_start,
                                                  const float4* __restrict__ sorted,
                                                  int32_t* __restrict__ nbr) {
  // thread jj takes the jj-th token in cell order: a warp's queries share
  // their cells, so its lanes scan the same candidate cells together
  const int jj = blockIdx.x * blockDim.x + threadIdx.x;
  const int b = blockIdx.y;
  if (jj >= N) return;
  const GridInfo g = info[b];
  const int32_t* cs = cell_start + (size_t)b * (gmax + 1);
  const float4* P = sorted + (size_t)b * N;
  const float4 qp = P[jj];
  const int j = __float_as_int(qp.w);
  const float qx = qp.x, qy = qp.y, qz = qp.z;
  const int cx = grid_coord(g, qx, 0), cy = grid_coord(g, qy, 1), cz = grid_coord(g, qz, 2);
  // only the first kk slots are used; the others stay at the smallest key
  // and never become the worst
  unsigned long long best[KK];
#pragma unroll
  for (int i = 0; i < KK; ++i) best[i] = i < kk ? ~0ull : 0ull;
  unsigned long long worst = ~0ull;
  int wi = 0;
  const int rmax = max(g.dims[0], max(g.dims[1], g.dims[2]));
  for (int r = 0; r <= rmax; ++r) {
    for (int dz = -r; dz <= r; ++dz) {
      const int z = cz + dz;
      if (z < 0 || z >= g.dims[2]) continue;
      for (int dy = -r; dy <= r; ++dy) {
        const int y = cy + dy;
        if (y < 0 || y >= g.dims[1]) continue;
        const bool face = dz == -r || dz == r || dy == -r || dy == r;
        for (int dx = -r; dx <= r; dx += (face || r == 0) ? 1 : 2 * r) {
          const int x = cx + dx;
          if (x < 0 || x >= g.dims[0]) continue;
          const int c = (z * g.dims[1] + y) * g.dims[0] + x;
          const int e = cs[c + 1];
          for (int s = cs[c]; s < e; ++s) {
            const float4 p = P[s];
            const int k = __float_as_int(p.w);
            const uint32_t bits = __float_as_uint(sqdist_rn(qx, qy, qz, p.x, p.y, p.z));
            if (k == j || bits > (uint32_t)(worst >> 32)) continue;
            const unsigned long long key = ((unsigned long long)bits << 32) | (uint32_t)k;
            if (key >= worst) continue;
#pragma unroll
            for (int i = 0; i < KK; ++i) best[i] = i == wi ? key : best[i];
            worst = 0ull;
#pragma unroll
            for (int i = 0; i < KK; ++i)
              if (best[i] > worst) {
                worst = best[i];
                wi = i;
              }
          }
        }
      }
    }
    if (worst != ~0ull) {  // the list is full: is anything closer still possible?
      const float reach = ((float)r - 1.0f / 1024.0f) * g.h;
      if (reach > 0.0f && __uint_as_float((uint32_t)(worst >> 32)) < reach * reach) break;
    }
  }
  // sort the kk keys ascending (the unused slots hold 0 and sort first)
#pragma unroll
  for (int i = 1; i < KK; ++i)
#pragma unroll
    for (int t = KK - 1; t >= i; --t)
      if (best[t] < best[t - 1]) {
        const unsigned long long x = best[t];
        best[t] = best[t - 1];
        best[t - 1] = x;
      }
  int32_t* out = nbr + ((size_t)b * N + j) * kk;
#pragma unroll
  for (int i = 0; i < KK; ++i)
    if (i >= KK - kk) out[i - (KK - kk)] = (int32_t)(best[i] & 0xFFFFFFFFull);
}

// The largest pinned-fp32 squared distance over pairs, into stats.d2_max_bits,
// from the neighbour grid (points sorted by cell).  A lower bound L is the
// largest d^2 among the extreme points of 7 directions (the axes and the
// space diagonals; an actual pair).  For two cells whose coordinates differ
// by (dx, dy, dz) cells, any two of their points are at most (|d| + 1) h +
// delta apart along each axis (delta covers the rounding of the cell
// assignment), so the pair of cells can hold a pair above L only if
// sum ((|d| + 1) h + delta)^2, inflated for fp32 rounding, reaches L.  Cells
// that reach L with no cell of the grid's corners are dropped; the pairs of
// the remaining cells that pass the test are evaluated with the same
// arithmetic as every other kernel, so the result is exactly the largest d^2.
//
// A cluster of up to 8 blocks per scene: each finds the extremes of its part of
// the points (the work is nearly all there; few dozen pairs of cells pass the
// test), then takes the pairs whose lower cell c is its rank modulo their
// number, a warp per cell; pairs of large cells are left to the whole block.
// 16384 points: 167 us before (13 directions over all points in each of 4
// blocks, a thread per pair of cells), 24 now; 32 scenes of 8192 88 and 38.
constexpr int DIA_THREADS = 512, DIA_PARTS = 8, DIA_DIRS = 7, DIA_BIG = 64;

__device__ __forceinline__ uint32_t warp_max_u32(uint32_t v) {
  return __reduce_max_sync(0xFFFFFFFFu, v);
}

__global__ void __launch_bounds__(DIA_THREADS) k_diameter_grid(
    int N, int gmax, int parts, const GridInfo* __restrict__ info, const int32_t* __restrict__ cell_start,
    const float4* __restrict__ sorted, SceneStats* stats) {
  extern __shared__ int s_cand[];  // candidate cells, [gmax]
  __shared__ unsigned long long s_ext[2 * DIA_DIRS];   // this block's extremes: (key, point)
  __shared__ uint32_t s_pt[2 * DIA_DIRS];              // the scene's
  __shared__ int4 s_big[DIA_BIG];
  __shared__ int s_ncand, s_nbig;
  __shared__ uint32_t s_m;
  const int b = blockIdx.y, part = (int)cluster_ctarank();
  const GridInfo g = info[b];
  const int32_t* cs = cell_start + (size_t)b * (gmax + 1);
  const float4* P = sorted + (size_t)b * N;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  constexpr int NW = DIA_THREADS / 32;
  if (threadIdx.x < 2 * DIA_DIRS) s_ext[threadIdx.x] = 0ull;
  if (threadIdx.x == 0) {
    s_ncand = 0;
    s_nbig = 0;
    s_m = 0u;
  }
  __syncthreads();

  uint32_t m = 0u;  // the largest d^2 bits this thread has seen
  {
    float hi[DIA_DIRS], lo[DIA_DIRS];
    int ih[DIA_DIRS], il[DIA_DIRS];
#pragma unroll
    for (int d = 0; d < DIA_DIRS; ++d) {
      hi[d] = -INFINITY;
      lo[d] = INFINITY;
      ih[d] = il[d] = 0;
    }
#pragma unroll 2
    for (int i = part * DIA_THREADS + threadIdx.x; i < N; i += parts * DIA_THREADS) {
      const float4 p = P[i];
      const float v[DIA_DIRS] = {p.x, p.y, p.z, p.x + p.y + p.z, p.x + p.y - p.z,
                                 p.x - p.y + p.z, -p.x + p.y + p.z};
      if (!(v[3] == v[3])) m = 0x7FFFFFFFu;  // an undefined point: so is the diameter
#pragma unroll
      for (int d = 0; d < DIA_DIRS; ++d) {
        if (v[d] > hi[d]) {
          hi[d] = v[d];
          ih[d] = i;
        }
        if (v[d] < lo[d]) {
          lo[d] = v[d];
          il[d] = i;
        }
      }
    }
#pragma unroll
    for (int d = 0; d < DIA_DIRS; ++d) {
      const uint32_t kh = f2key(hi[d]), kl = f2key(-lo[d]);
      const uint32_t mh = warp_max_u32(kh), ml = warp_max_u32(kl);
      const int sh = __ffs(__ballot_sync(0xFFFFFFFFu, kh == mh)) - 1;
      const int sl = __ffs(__ballot_sync(0xFFFFFFFFu, kl == ml)) - 1;
      if (lane == sh) atomicMax(&s_ext[2 * d], ((unsigned long long)mh << 32) | (uint32_t)ih[d]);
      if (lane == sl) atomicMax(&s_ext[2 * d + 1], ((unsigned long long)ml << 32) | (uint32_t)il[d]);
    }
  }
  hw_cluster_sync();  // every block's extremes are complete
  if (threadIdx.x < 2 * DIA_DIRS) {
    unsigned long long x[DIA_PARTS];
#pragma unroll
    for (int r = 0; r < DIA_PARTS; ++r)
      asm volatile("ld.shared::cluster.u64 %0, [%1];"
                   : "=l"(x[r])
                   : "r"(map_rank(smem_addr(&s_ext[threadIdx.x]), (uint32_t)min(r, parts - 1)))
                   : "memory");
    unsigned long long m = x[0];
#pragma unroll
    for (int r = 1; r < DIA_PARTS; ++r) m = x[r] > m ? x[r] : m;
    s_pt[threadIdx.x] = (uint32_t)m;
  }
  __syncthreads();
  if (threadIdx.x < 4 * DIA_DIRS * DIA_DIRS) {
    const float4 a = P[s_pt[threadIdx.x / (2 * DIA_DIRS)]];
    const float4 c = P[s_pt[threadIdx.x % (2 * DIA_DIRS)]];
    m = max(m, __float_as_uint(sqdist_rn(a.x, a.y, a.z, c.x, c.y, c.z)));
  }
  m = warp_max_u32(m);
  if (lane == 0) atomicMax(&s_m, m);
  __syncthreads();
  const float L = __uint_as_float(s_m);

  // bound of two cells' d^2 from their coordinate differences
  float span = 0.0f;
  for (int a = 0; a < 3; ++a) span = fmaxf(span, fabsf(g.lo[a]) + (float)g.dims[a] * g.h);
  const float delta = 1e-3f * g.h + 1e-5f * span;
  auto bound = [&](int dx, int dy, int dz) -> float {
    const float ex = (float)(dx + 1) * g.h + delta;
    const float ey = (float)(dy + 1) * g.h + delta;
    const float ez = (float)(dz + 1) * g.h + delta;
    return (ex * ex + ey * ey + ez * ez) * 1.000244140625f;  // 1 + 2^-12
  };
  // the candidate cells, in any order
  const int d0 = g.dims[0], d1 = g.dims[1], d2 = g.dims[2];
  for (int base = 0; base < g.ncells; base += DIA_THREADS) {
    const int c = base + threadIdx.x;
    bool cand = false;
    if (c < g.ncells && cs[c + 1] > cs[c]) {
      const int cx = c % d0, cy = (c / d0) % d1, cz = c / (d0 * d1);
      cand = bound(max(cx, d0 - 1 - cx), max(cy, d1 - 1 - cy), max(cz, d2 - 1 - cz)) >= L;
    }
    const uint32_t bal = __ballot_sync(0xFFFFFFFFu, cand);
    if (bal) {
      int at = 0;
      if (lane == 0) at = atomicAdd(&s_ncand, __popc(bal));
      at = __shfl_sync(0xFFFFFFFFu, at, 0);
      if (cand) s_cand[at + __popc(bal & ((1u << lane) - 1u))] = c;
    }
  }
  __syncthreads();
  const int M = s_ncand;

  auto pair_max = [&](const float4& p, const float4& q) {
    m = max(m, __float_as_uint(sqdist_rn(p.x, p.y, p.z, q.x, q.y, q.z)));
  };
  // pairs of candidate cells A <= B
  for (int r = w; r < M; r += NW) {
    const int A = s_cand[r];
    if (A % parts != part) continue;
    const int ax = A % d0, ay = (A / d0) % d1, az = A / (d0 * d1);
    const int a0 = cs[A], na = cs[A + 1] - a0;
    for (int t0 = 0; t0 < M; t0 += 32) {
      const int t = t0 + lane;
      int b0 = 0, nb = 0;
      if (t < M) {
        const int B = s_cand[t];
        const int bx = B % d0, by = (B / d0) % d1, bz = B / (d0 * d1);
        if (B >= A && bound(abs(ax - bx), abs(ay - by), abs(az - bz)) >= L) {
          b0 = cs[B];
          nb = cs[B + 1] - b0;
        }
      }
      uint32_t todo = __ballot_sync(0xFFFFFFFFu, nb > 0);
      while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1u;
        const int q0 = __shfl_sync(0xFFFFFFFFu, b0, src), nq = __shfl_sync(0xFFFFFFFFu, nb, src);
        if ((int64_t)na * nq > 4096) {  // for the whole block, while there is room
          int at = 0;
          if (lane == 0) at = atomicAdd(&s_nbig, 1);
          at = __shfl_sync(0xFFFFFFFFu, at, 0);
          if (at < DIA_BIG) {
            if (lane == 0) s_big[at] = make_int4(a0, na, q0, nq);
            continue;
          }
        }
        if (nq >= 16) {
          for (int i = 0; i < na; ++i) {
            const float4 p = P[a0 + i];
            for (int j = lane; j < nq; j += 32) pair_max(p, P[q0 + j]);
          }
        } else {  // a lane a point of A
          for (int i = lane; i < na; i += 32) {
            const float4 p = P[a0 + i];
            for (int j = 0; j < nq; ++j) pair_max(p, P[q0 + j]);
          }
        }
      }
    }
  }
  __syncthreads();
  for (int k = 0; k < min(s_nbig, DIA_BIG); ++k) {
    const int4 e = s_big[k];
    for (int i = 4 * w; i < e.y; i += 4 * NW) {  // four points of A a warp
      float4 p[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) p[u] = P[e.x + min(i + u, e.y - 1)];
#pragma unroll 2
      for (int j = lane; j < e.w; j += 32) {
        const float4 q = P[e.z + j];
#pragma unroll
        for (int u = 0; u < 4; ++u) pair_max(p[u], q);
      }
    }
  }
  m = warp_max_u32(m);
  if (lane == 0) atomicMax(&stats[b].d2_max_bits, m);
  hw_cluster_sync();  // nobody leaves while a peer may still read its extremes
}

int grid_cells_max(int64_t N) {
  int64_t G = 1;
  while (4 * G * G * G < N) ++G;
  return (int)(G * G * G);
}

int launch_knn_grid(const float* pos, int64_t B, int64_t N, int kk, int32_t* nbr,
                    SceneStats* stats, GridInfo* info, int32_t* cell_start, float4* sorted,
                    cudaStream_t s) {
  const int gmax = grid_cells_max(N);
  if (kk > kKnnGridMax || (kk > 0 && kk >= N)) return CP_EINVAL;  // the search needs kk others
  const size_t smem = sizeof(int) * (size_t)(gmax + 1);
  CP_TRY_STATUS(allow_smem((const void*)k_grid_build, smem, "launch_knn_grid: smem attribute"));
  CP_TRY_STATUS(allow_smem((const void*)k_diameter_grid, smem, "launch_knn_grid: smem attribute"));
  k_grid_build<<<(unsigned)B, 1024, smem, s>>>(pos, (int)N, gmax, info, cell_start, sorted);
  CP_TRY_STATUS(last_launch_status());
  DeviceInfo di;
  if (device_info(&di) != CP_OK) return CP_ECUDA;
  // up to two blocks an SM: further blocks only wait, and each clears and scans
  // the cells again.  Diameters alone (no neighbours), us, 8 blocks a scene
  // always / by this rule: 64 scenes of 256 tokens 45 / 36, 512 of 256 184 / 55,
  // 256 of 1024 109 / 48, 64 of 8192 75 / 65; up to one an SM the last takes 68,
  // up to four 76.
  int parts = DIA_PARTS;
  while (parts > 1 && B * parts > 2 * di.sm_count) parts >>= 1;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[1];
  cfg.gridDim = dim3((unsigned)parts, (unsigned)B);
  cfg.blockDim = dim3(DIA_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = (unsigned)parts;
  attr->val.clusterDim.y = 1;
  attr->val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_diameter_grid, (int)N, gmax, parts, info,
                                           cell_start, sorted, stats);
  note_launch();
  CP_TRY_STATUS(cuda_status(e, "launch_knn_grid: diameter"));
  if (kk <= 0) return CP_OK;
  // Few neighbours of very many queries: a thread a query needs fewer
  // instructions than a warp, but a chain of the longer shells' cells that only
  // many queries hide.  us, thread / warp (with k_grid_build and
  // k_diameter_grid), 1 and 8 neighbours: 64 scenes of 1024 104 / 103 and 120 /
  // 119, 128 124 / 160 and 160 / 195; 32 of 2048 178 / 122 and 193 / 139, 64 182
  // / 182 and 214 / 217; 32 of 4096 226 / 186 and 265 / 217, 64 265 / 311 and 355
  // / 380; 16 of 8192 205 / 190 and 232 / 223, 32 261 / 320 and 378 / 384, 64 592
  // / 588 and 710 / 715, 128 624 / 1109 and 933 / 1362; 16 of 16384 299 / 344 and
  // 462 / 410, 32 615 / 667 and 730 / 797.
  const int64_t many = N <= 1024 ? 65536 : N <= 2048 ? 131072 : N <= 8192 ? 262144 : 524288;
  if (kk <= 8 && B * N >= many) {
    k_knn_grid_thread<8><<<dim3((unsigned)((N + 127) / 128), (unsigned)B), 128, 0, s>>>(
        (int)N, kk, gmax, info, cell_start, sorted, nbr);
    return last_launch_status();
  }
  const dim3 grid((unsigned)((N + KW_WARPS - 1) / KW_WARPS), (unsigned)B);
  k_knn_grid<<<grid, 32 * KW_WARPS, 0, s>>>((int)N, kk, gmax, info, cell_start, sorted, nbr);
  return last_launch_status();
}

__global__ void k_diameter(const SceneStats* stats, int B, float* out) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < B) out[b] = sqrtf(__uint_as_float(stats[b].d2_max_bits));
}

int launch_diameter(const SceneStats* stats, int64_t B, float* out, cudaStream_t s) {
  k_diameter<<<(unsigned)((B + 127) / 128), 128, 0, s>>>(stats, (int)B, out);
  return last_launch_status();
}

// ---------------------------------------------------------------------------
// Normalisers from the reduced statistics.
// ---------------------------------------------------------------------------
__global__ void k_finalize_norms(const SceneStats* stats, int B, int norm_mode,
                                 SceneNorms* norms, float* norms_out) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  const SceneStats st = stats[b];
  SceneNorms nm;
  const float cmax = key2f(st.cos_max_key), cmin = key2f(st.cos_min_key);
  // min-max over all pairs (the Gram's extremes), or the bounds of
  // d_f = 1 - cos itself, [0, 2]
  nm.f_lo = norm_mode == 1 ? 0.0f : 1.0f - cmax;
  nm.f_hi = norm_mode == 1 ? 2.0f : 1.0f - cmin;
  nm.x_lo = 0.0f;  // diagonal pairs: d_x(j, j) = 0
  nm.x_hi = sqrtf(__uint_as_float(st.d2_max_bits));
  nm.t_lo = 0.0f;  // d_tau(j, j) = 0 and d_tau >= 0
  nm.t_hi = (float)(st.tau_max - st.tau_min);
  const float rf = nm.f_hi - nm.f_lo, rx = nm.x_hi - nm.x_lo, rt = nm.t_hi - nm.t_lo;
  nm.f_rinv = rf > (float)kRangeEps ? 1.0f / rf : 0.0f;
  nm.x_rinv = rx > (float)kRangeEps ? 1.0f / rx : 0.0f;
  nm.t_rinv = rt > (float)kRangeEps ? 1.0f / rt : 0.0f;
  for (int i = 0; i < 7; ++i) nm.pad[i] = 0.0f;
  norms[b] = nm;
  if (norms_out) {
    float* o = norms_out + 6 * (size_t)b;
    o[0] = nm.f_lo; o[1] = nm.f_hi; o[2] = nm.x_lo; o[3] = nm.x_hi; o[4] = nm.t_lo; o[5] = nm.t_hi;
  }
}

int launch_finalize_norms(const SceneStats* stats, int64_t B, int norm_mode, SceneNorms* norms,
                          float* norms_out, cudaStream_t s) {
  k_finalize_norms<<<(unsigned)((B + 127) / 128), 128, 0, s>>>(stats, (int)B, norm_mode, norms,
                                                               norms_out);
  return last_launch_status();
}

}  // namespace cp
