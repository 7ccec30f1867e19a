// K5, the default greedy selection (sgs_mode 0): every candidate's exact gain
// is kept up to date, so a step is an argmax and a few list updates.
//
// A term v_j max(m_j - C(t, j), 0) of gain(t) can only change when a pick
// lowers m_j, and it is zero for good once C(t, j) >= m_j.  So every target j
// keeps the list of its live candidates -- the (t, C(t, j)) with C(t, j) <
// m_j -- and a pick w that lowers m_j from a to b takes
//     term(v_j, a, C(t, j)) - term(v_j, b, C(t, j))
// off the gain of each t on j's list and drops the entries with C(t, j) >= b.
// Terms are fixed-point integers (sgs_gain.cuh), so the kept gains equal the
// gains summed afresh, bit for bit, whatever order the updates ran in.
//
// The lists are short: on the dense path they are formed once the first pick
// is known (k_live_lists, one pass over the cost), when about a fifth to a
// quarter of all pairs is still live (long video 0.21, short clip 0.27 of
// N^2); a whole selection of a long-video scene (N = 8192, K = 1229) then
// touches 21 M entries, and steps past 410 change ~8 targets and ~150
// entries.  On the local path the live candidates of j start as the t with j
// in M_g(t) (k_rev_fill).
//
// The work is little; what bounds it is chains of dependent latencies --
// argmax, the winner's row, the lowered targets' lists, the gain updates --
// with block barriers between.  Two kernels share the steps:
//  - k_sgs_push, one pick a step, while a pick lowers many targets (dense
//    path): a cluster of blocks per scene, ~2 us a step;
//  - k_sgs_rounds, one block per scene, many picks a round, for the rest
//    (and all of a local selection): late picks lower few targets each,
//    mostly different ones, so dozens of them are independent of one another.
// Selection of 1229 of 8192 tokens: 2.7 ms (re-evaluating candidate rows
// behind bounds, the approach before these: 11.9; one pick a step to the end:
// 5.9); 410 of 4096: 1.05 (3.8, 2.1); 32 scenes of 8192: 8.5 (19.9, 12.0).
#include <string.h>

#include "bf16_dot.cuh"
#include "sgs_gain.cuh"

namespace cp {
namespace {

constexpr int PUSH_CMAX = 16;  // blocks per cluster (16: the non-portable maximum)
constexpr int PUSH_WARPS = 32;
// The single-pick steps end once the running mean of the targets a pick
// lowers is below this: a step costs ~2 us whatever it lowers, a pick of a
// round costs its lists' share of one block, and where rows are still longer
// than RD_ROW rounds pick one at a time.  Selection, ms, with a warp a list,
// at 16 / 24 / 32 / 40 / 48 / 64: N = 1024 0.34 / 0.32 / 0.32 / 0.31 / 0.31 /
// 0.30, N = 4096 1.22 / 1.20 / 1.15 / 1.14 / 1.13 / 1.12, N = 8192 3.00 / 2.97
// / 2.96 / 2.95 / 3.22 / 3.21, 32 scenes of N = 8192 8.65 / 8.52 / 8.54 / 8.61
// / 9.17 / 9.23.
constexpr int PUSH_STOP = 36;
constexpr int PUSH_THREADS = 32 * PUSH_WARPS;

// 8 bytes into another block's shared memory, counted on the mbarrier there
// (both addresses mapped to that block).
__device__ __forceinline__ void st_async_u64(uint32_t dst, gain_t v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.u64 [%0], %1, [%2];" ::"r"(
                   dst),
               "l"(v), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// One live candidate of a target: the candidate's index in its owner block
// and its cost bits.
typedef uint2 Entry;

// ---------------------------------------------------------------------------
// The first pick of the dense path.  The cost pass's partial sums (g0, one
// per 64-column tile) add the gain's terms in fp32: at most 8 roundings
// inside a tile and one per tile after that, each of relative size 2^-24 of
// non-negative sums, so a total is within 2^-15 (264 x 2^-24 at 256 tiles)
// of the exact sum, the fixed-point gain (two roundings a term) and its 24
// bits among the 248 x 2^-24 to spare.  Only candidates whose upper bound
// reaches the largest lower bound can be the first pick; their gains are
// computed exactly.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_first_bounds(const float* __restrict__ g0, int slots, int N,
                                                      float* __restrict__ sums,
                                                      uint32_t* __restrict__ max_bits) {
  const int t = blockIdx.x * 256 + threadIdx.x, b = blockIdx.y;
  float sum = 0.0f;
  if (t < N) {
    const float* p = g0 + (size_t)b * slots * N + t;
#pragma unroll 16
    for (int sl = 0; sl < slots; ++sl) sum += __ldg(p + (size_t)sl * N);
    sum = fmaxf(sum, 0.0f);
    sums[(size_t)b * N + t] = sum;
  }
  const uint32_t m = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(sum));
  if ((threadIdx.x & 31) == 0) atomicMax(max_bits + b, m);
}

// Exact gains at m = m0 of the candidates that may be the first pick (all of
// them without bounds); the best key by atomicMax.  A warp scans 32
// candidates' bounds at a time and evaluates the ones that pass.
__global__ void __launch_bounds__(256) k_first_pick(const float* __restrict__ cost, int64_t ldc,
                                                    const float* __restrict__ v_all,
                                                    int N, float m0, int fx,
                                                    const float* __restrict__ sums,
                                                    const uint32_t* __restrict__ max_bits,
                                                    gain_t* __restrict__ first) {
  const int b = blockIdx.y, lane = threadIdx.x & 31;
  const int gw = blockIdx.x * 8 + (threadIdx.x >> 5), nw = gridDim.x * 8;
  const float* v = v_all + (size_t)b * N;
  const float4* C4 = reinterpret_cast<const float4*>(cost + (size_t)b * N * ldc);
  const int nq = (int)(ldc >> 2);
  const float least = sums ? __uint_as_float(max_bits[b]) * 0.999969482421875f : 0.0f;  // 1 - 2^-15
  gain_t best = 0ull;
  // candidates in groups of 32 dealt round-robin over the warps: with bounds
  // few pass; without them a warp takes one candidate at a time
  const int span = sums ? 32 : 1;
  for (int t0 = gw * span; t0 < N; t0 += nw * span) {
    const int t = t0 + lane;
    bool pass = lane < span && t < N;
    if (pass && sums) pass = sums[(size_t)b * N + t] * 1.000030517578125f >= least;  // 1 + 2^-15
    uint32_t todo = __ballot_sync(0xFFFFFFFFu, pass);
    while (todo) {
      const int tc = t0 + __ffs(todo) - 1;
      todo &= todo - 1u;
      const float4* row = C4 + (size_t)tc * nq;
      gain_t acc = 0ull;
      for (int i0 = lane; i0 - lane < nq; i0 += 8 * 32) {
        float4 c[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          c[u] = i0 + 32 * u < nq ? ld_stream_f4(row + i0 + 32 * u) : make_float4(m0, m0, m0, m0);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int j = 4 * (i0 + 32 * u);
          const float cc[4] = {c[u].x, c[u].y, c[u].z, c[u].w};
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (j + e < N) acc += gain_term(__ldg(v + j + e), m0, cc[e], fx);
        }
      }
      const gain_t key = gain_key(gain_bits(warp_sum_gain(acc), fx), tc);
      best = key > best ? key : best;
    }
  }
  if (lane == 0 && best) atomicMax(first + b, best);
}

// The scale after the first pick where m0's and the largest cost's differ: m0's
// while a target is still uncovered (its cost undefined, as of a token with an
// infinite coordinate).
__global__ void __launch_bounds__(256) k_first_scale(const float* __restrict__ cost, int64_t ldc,
                                                     const gain_t* __restrict__ first, int N,
                                                     float m0, int fx0, int fx,
                                                     int* __restrict__ fxs) {
  const int b = blockIdx.x;
  const float* row = cost + ((size_t)b * N + key_token(first[b])) * ldc;
  bool open = false;
  for (int j = threadIdx.x; j < N; j += 256) open |= !(__ldg(row + j) < m0);
  open = __syncthreads_or(open);
  if (threadIdx.x == 0) fxs[b] = open ? fx0 : fx;
}

// ---------------------------------------------------------------------------
// The live candidates after the first pick w0, m_j = min(m0, C(w0, j)), and
// every candidate's gain there: one pass over the cost.  A block owns 128
// columns of one owner's rows (t = tl C + rank): tiles of 32 rows x 128
// columns come in by cp.async, four deep; a warp takes 8 of the columns with
// a lane per row (one 16-byte shared load covers four columns), so a
// column's live rows are one ballot, the entries of a list go out
// contiguously and a lane's gain needs no reduction until the tile ends.
// Candidates with nearby indices are near in space, so about half of the
// ballots are empty and skip the arithmetic.  32 scenes of N = 8192: 2.7 ms,
// 4.8 TB/s of reads (8.6 GB, the cost once) and writes (8 bytes a live entry,
// 4.2 GB); bound by instruction issue before HBM: a column of a tile costs its
// ballot, a live one its term and store besides.
// List of (j, owner): lists[((bl N + j) C + owner) NC ..], lens alike.
// ---------------------------------------------------------------------------
constexpr int LL_COLS = 128, LL_ROWS = 32, LL_STAGES = 4, LL_WARPS = 16;
constexpr int LL_PITCH = LL_COLS + 4;  // lanes of a 16-byte read (a lane a row) on distinct banks
constexpr int LL_COLS_W = LL_COLS / LL_WARPS;
constexpr size_t LL_SMEM = sizeof(float) * LL_STAGES * LL_ROWS * LL_PITCH;

template <bool SCALED>  // the scene's scale is fxs[b]
__global__ void __launch_bounds__(32 * LL_WARPS) k_live_lists(
    const float* __restrict__ cost, int64_t ldc, const float* __restrict__ v_all,
    const gain_t* __restrict__ first, int N, int C, int lgC, int NC, int scene0, float m0,
    int fx_all, const int* __restrict__ fxs, gain_t* __restrict__ gains,
    Entry* __restrict__ lists, uint32_t* __restrict__ lens) {
  extern __shared__ __align__(16) float s_tile[];  // [LL_STAGES][LL_ROWS][LL_PITCH]
  __shared__ gain_t s_part[2][LL_WARPS][32];
  const int col0 = blockIdx.x * LL_COLS, rank = blockIdx.y, bl = blockIdx.z, b = scene0 + bl;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float* Cb = cost + (size_t)b * N * ldc;
  const float* v = v_all + (size_t)b * N;
  gain_t* G = gains + (size_t)b * N;
  const int fx = SCALED ? __ldg(fxs + b) : fx_all;
  const int nown = N > rank ? (N - rank + C - 1) >> lgC : 0;
  const int ntile = (nown + LL_ROWS - 1) / LL_ROWS;
  const int w0 = key_token(first[b]);
  const uint32_t lstep = (uint32_t)(C * NC);  // between the lists of adjacent columns
  float m[LL_COLS_W], vj[LL_COLS_W];
  uint32_t pos[LL_COLS_W];   // the column's next free entry, from the warp's first list
#pragma unroll
  for (int u = 0; u < LL_COLS_W; ++u) {
    const int j = col0 + LL_COLS_W * w + u;
    m[u] = -INFINITY;  // past the row: nothing is live
    vj[u] = 0.0f;
    pos[u] = (uint32_t)u * lstep;
    if (j < N) {
      m[u] = fminf(m0, __ldg(Cb + (size_t)w0 * ldc + j));
      vj[u] = __ldg(v + j);
    }
  }
  Entry* L = lists + ((size_t)((size_t)bl * N + col0 + LL_COLS_W * w) * C + rank) * NC;
  auto load = [&](int i) {
    float* dst = s_tile + (size_t)(i % LL_STAGES) * LL_ROWS * LL_PITCH;
#pragma unroll
    for (int q = 0; q < LL_ROWS * (LL_COLS / 4) / (32 * LL_WARPS); ++q) {
      const int idx = threadIdx.x + 32 * LL_WARPS * q;
      const int r = idx / (LL_COLS / 4), c4 = 4 * (idx % (LL_COLS / 4));
      const int tl = LL_ROWS * i + r;
      const bool ok = tl < nown && col0 + c4 < ldc;  // ldc % 4 == 0
      const float* src = ok ? Cb + (size_t)((tl << lgC) | rank) * ldc + col0 + c4 : Cb;
      cp_async16_zfill(dst + r * LL_PITCH + c4, src, ok);
    }
  };
  // the 16 warps' partial gains of tile i's rows, added to the scene's
  auto flush = [&](int i) {
    gain_t s = 0ull;
#pragma unroll
    for (int q = 0; q < LL_WARPS; ++q) s += s_part[i & 1][q][lane];
    const int tl = LL_ROWS * i + lane;
    if (s != 0ull && tl < nown) atomicAdd(G + ((tl << lgC) | rank), s);
  };
#pragma unroll
  for (int i = 0; i < LL_STAGES - 1; ++i) {
    if (i < ntile) load(i);
    cp_commit();
  }
  const uint32_t lt = (1u << lane) - 1u;
  for (int i = 0; i < ntile; ++i) {
    cp_wait<LL_STAGES - 2>();
    __syncthreads();  // tile i is in; tile i - 1 and its partial gains are complete
    if (i + LL_STAGES - 1 < ntile) load(i + LL_STAGES - 1);  // over tile i - 1's stage
    cp_commit();
    if (i > 0 && w == ((i - 1) & (LL_WARPS - 1))) flush(i - 1);
    const float* tile = s_tile + (size_t)(i % LL_STAGES) * LL_ROWS * LL_PITCH +
                        lane * LL_PITCH + LL_COLS_W * w;
    const int tl = LL_ROWS * i + lane;
    const bool row_ok = tl < nown;
    gain_t acc = 0ull;
#pragma unroll
    for (int h = 0; h < LL_COLS_W / 4; ++h) {
      const float4 c4 = *reinterpret_cast<const float4*>(tile + 4 * h);
      const float c[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int u = 4 * h + e;
        const bool live = row_ok && c[e] < m[u];
        const uint32_t mask = __ballot_sync(0xFFFFFFFFu, live);
        if (mask) {  // warp-uniform
          if (live) {
            acc += gain_term(vj[u], m[u], c[e], fx);
            L[pos[u] + __popc(mask & lt)] = make_uint2((uint32_t)tl, __float_as_uint(c[e]));
          }
          pos[u] += __popc(mask);
        }
      }
    }
    s_part[i & 1][w][lane] = acc;
  }
  __syncthreads();
  if (ntile > 0 && w == ((ntile - 1) & (LL_WARPS - 1))) flush(ntile - 1);
  if (lane == 0) {
#pragma unroll
    for (int u = 0; u < LL_COLS_W; ++u) {
      const int j = col0 + LL_COLS_W * w + u;
      if (j < N) lens[((size_t)bl * N + j) * C + rank] = pos[u] - (uint32_t)u * lstep;
    }
  }
}

// ---------------------------------------------------------------------------
// The local path's lists: the candidates t with j in M_g(t) and their costs.
// Counts (a warp a candidate), an exclusive scan (a block a scene) and the
// fill, which also sums the candidates' first gains (m = m0).  span[b N + j] =
// (offset into the scene's entries, length); the order within a list is
// arbitrary (no result depends on it).  Bound by L2 atomics: 4 scenes of
// 6272, g = 64, 63 us (one block a scene doing all of it: 489), 32 of 8192
// 419 (728).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_rev_count(const int32_t* __restrict__ nbr, int N, int g,
                                                   int kk, uint2* __restrict__ span) {
  const int t = blockIdx.x * 8 + (threadIdx.x >> 5), b = blockIdx.y, lane = threadIdx.x & 31;
  if (t >= N) return;
  const int32_t* nb = nbr + ((size_t)b * N + t) * kk;
  for (int k = lane; k < g; k += 32)
    atomicAdd(&span[(size_t)b * N + (k == 0 ? t : __ldg(nb + k - 1))].y, 1u);
}

__global__ void __launch_bounds__(1024) k_rev_scan(int N, uint2* __restrict__ span_all) {
  __shared__ uint32_t s_w[32];
  uint2* span = span_all + (size_t)blockIdx.x * N;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint32_t carry = 0u;
  for (int j0 = 0; j0 < N; j0 += 4096) {  // four a thread
    const int j = j0 + 4 * (int)threadIdx.x;
    uint32_t n[4], sum = 0u;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      n[u] = j + u < N ? span[j + u].y : 0u;
      sum += n[u];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += x;
    }
    __syncthreads();  // the last turn's sums are read
    if (lane == 31) s_w[w] = incl;
    __syncthreads();
    const uint32_t x = s_w[lane];
    uint32_t run = carry + __reduce_add_sync(0xFFFFFFFFu, lane < w ? x : 0u) + incl - sum;
    carry += __reduce_add_sync(0xFFFFFFFFu, x);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (j + u < N) span[j + u] = make_uint2(run, 0u);  // the fill counts again
      run += n[u];
    }
  }
}

__global__ void __launch_bounds__(256) k_rev_fill(const float* __restrict__ slab,
                                                  const int32_t* __restrict__ nbr,
                                                  const float* __restrict__ v_all, int N, int g,
                                                  int kk, float m0, int fx,
                                                  uint2* __restrict__ span_all,
                                                  Entry* __restrict__ ent_all,
                                                  gain_t* __restrict__ gains) {
  const int t = blockIdx.x * 8 + (threadIdx.x >> 5), b = blockIdx.y, lane = threadIdx.x & 31;
  if (t >= N) return;
  const float* v = v_all + (size_t)b * N;
  const float* srow = slab + ((size_t)b * N + t) * g;
  const int32_t* nb = nbr + ((size_t)b * N + t) * kk;
  uint2* span = span_all + (size_t)b * N;
  Entry* ent = ent_all + (size_t)b * N * g;
  gain_t acc = 0ull;
  for (int k = lane; k < g; k += 32) {
    const int j = k == 0 ? t : __ldg(nb + k - 1);
    const float c = __ldg(srow + k);
    const uint32_t at = atomicAdd(&span[j].y, 1u);
    ent[span[j].x + at] = make_uint2((uint32_t)t, __float_as_uint(c));
    acc += gain_term(__ldg(v + j), m0, c, fx);
  }
  acc = warp_sum_gain(acc);
  if (lane == 0) gains[(size_t)b * N + t] = acc;
}

// ---------------------------------------------------------------------------
// The greedy steps while picks lower many targets (dense path): one pick a
// step.  Nothing in a step needs more than one SM but the long lists, so a
// scene runs on a small cluster of blocks: block r of C owns the candidates
// t = r (mod C) with their gains and its own part of every list, keeps its
// own copy of m, and per step exchanges one key with the others (st.async
// into every block's slot, counted on an mbarrier there: ~450 cycles, about
// a fifth of a late step; a barrier of the cluster takes twice that).
// ---------------------------------------------------------------------------
struct PushArgs {
  const float* cost;      // [B][N][ldc]
  const float* v;         // [B][N]
  gain_t* gains;          // [B][N] gains at the start; at the end the current ones
  const gain_t* first;    // [B] key of the first pick
  Entry* lists;
  uint32_t* lens;         // [scenes of the wave][N][C]
  float* m_out;           // [scenes of the wave][N] coverage cost where the steps stopped
  int* stop;              // [scenes of the wave] first step not taken
  int32_t* order32;       // [B][K]
  float* out_gains;       // [B][K] or null
  int* status;
  int64_t ldc;
  uint64_t timeout_ns;
  const int* fxs;         // [B] the scenes' scales, or null: fx
  float m0;
  int fx;
  int N, K;
  int C, lgC, NC;         // blocks per cluster (a power of two), its log2, ceil(N / C)
  int lgS;                // log2 of the candidates a warp scans
  int scene0;             // first scene of the wave
  uint32_t off_q, off_lo, off_hi;  // dynamic shared memory offsets
};

// One live candidate of a target lowered from mo to mn: its gain loses what
// the drop took.  Gains are kept as two 32-bit words (32-bit shared atomics
// are native): the low word's update goes out first and `old` carries what it
// saw, so that chunk_high, called once the low words of all entries in flight
// are on their way, takes the borrow off the high word; the pair is right once
// every update has run.
__device__ __forceinline__ gain_t chunk_low(uint32_t* lo, uint32_t at, float v, float mo, float mn,
                                            float c, int fx, uint32_t& old) {
  const gain_t d = gain_drop(v, mo, mn, c, fx);
  old = 0u;
  if (d != 0ull) old = atomicAdd(lo + at, 0u - (uint32_t)d);
  return d;
}
__device__ __forceinline__ void chunk_high(uint32_t* hi, uint32_t at, gain_t d, uint32_t old) {
  if (d != 0ull) {
    const uint32_t dh = (uint32_t)(d >> 32) + (old < (uint32_t)d ? 1u : 0u);
    if (dh) atomicAdd(hi + at, 0u - dh);
  }
}
template <int LW, bool SCALED = false>
__global__ void __launch_bounds__(PUSH_THREADS, 1) k_sgs_push(const __grid_constant__ PushArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  float* sm_m = reinterpret_cast<float*>(smem);                     // [ldc] coverage cost
  uint32_t* queue = reinterpret_cast<uint32_t*>(smem + a.off_q);    // [N] lowered targets
  uint32_t* g_lo = reinterpret_cast<uint32_t*>(smem + a.off_lo);    // [NC] gains, low words
  uint32_t* g_hi = reinterpret_cast<uint32_t*>(smem + a.off_hi);    // [NC] ... and high words
  __shared__ gain_t s_key[PUSH_WARPS];   // best key of each warp's candidates
  __shared__ uint32_t s_dirty[PUSH_WARPS];  // ... which of them changed since
  __shared__ gain_t s_res[2][PUSH_CMAX];    // exchanged keys, by step parity
  __shared__ __align__(8) uint64_t s_bar[2];
  __shared__ int s_qn, s_fail;

  const int rank = (int)cluster_ctarank();
  const int bl = (int)(blockIdx.x >> a.lgC), b = a.scene0 + bl;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int N = a.N, lgC = a.lgC, fx = SCALED ? __ldg(a.fxs + b) : a.fx;
  const int ncols = (int)a.ldc;
  const int nown = N > rank ? (N - rank + a.C - 1) >> lgC : 0;
  const float* v = a.v + (size_t)b * N;
  const float* R = a.cost + (size_t)b * N * (size_t)a.ldc;
  uint32_t my_ent = 0u;  // list entries read (a list's first lane counts; at most N^2 < 2^32)

  // state at the start: the first pick, m and the gains
  const gain_t f0 = a.first[b];
  int last = key_token(f0);  // the last pick, not yet dropped from the candidates
  if (rank == 0 && threadIdx.x == 0) {
    a.order32[(size_t)b * a.K] = last;
    if (a.out_gains) a.out_gains[(size_t)b * a.K] = key_gain(f0);
  }
  for (int j = threadIdx.x; j < ncols; j += PUSH_THREADS)
    sm_m[j] = j < N ? fminf(a.m0, __ldg(R + (size_t)last * a.ldc + j)) : 0.0f;
  for (int tl = threadIdx.x; tl < nown; tl += PUSH_THREADS) {
    const gain_t x = a.gains[(size_t)b * N + ((tl << lgC) | rank)];
    g_lo[tl] = (uint32_t)x;
    g_hi[tl] = (uint32_t)(x >> 32);
  }
  if (threadIdx.x < PUSH_WARPS) s_dirty[threadIdx.x] = 1u;
  if (threadIdx.x == 0) {
    s_qn = 0;
    s_fail = 0;
    mbar_init(&s_bar[0], 1);
    mbar_init(&s_bar[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  hw_cluster_sync();  // every block initialised before any peer writes to it
  const int lo0 = w << a.lgS, lo1 = min(nown, lo0 + (1 << a.lgS));  // this warp's candidates

  const uint32_t low = gain_floor(fx);
  bool ok = true;
  int pref = -1;  // the row last prefetched
  int step = 1;
  int mean8 = N;  // 8 x the running mean of the lowered targets a step
  for (; step < a.K && mean8 > 8 * PUSH_STOP; ++step) {
    const int par = step & 1;
    if (a.C > 1 && threadIdx.x == 0) mbar_expect(&s_bar[par], 8u * (uint32_t)a.C);
    // ---- the warp's best key, when one of its gains changed
    const int ltl = last >> lgC;
    const bool drop = (last & (a.C - 1)) == rank && ltl >= lo0 && ltl < lo1;
    if (drop || s_dirty[w] != 0u) {
      if (drop && lane == 0) g_hi[ltl] = 0xFFFFFFFFu;  // selected: no candidate any more
      __syncwarp();
      if (lane == 0) s_dirty[w] = 0u;
      uint32_t bf = 0u;
      int bt = 0x7FFFFFFF;
      for (int tl = lo0 + lane; tl < lo1; tl += 32) {
        const uint32_t hi = g_hi[tl];
        const gain_t x = ((gain_t)hi << 32) | g_lo[tl];
        const uint32_t f = (int)hi < 0 ? 0u : gain_bits(x, fx) + 1u;
        if (f > bf) {  // ascending tl: the lowest index among equals stays
          bf = f;
          bt = tl;
        }
      }
      const uint32_t mf = __reduce_max_sync(0xFFFFFFFFu, bf);
      const int mt = __reduce_min_sync(0xFFFFFFFFu, bf == mf ? bt : 0x7FFFFFFF);
      if (lane == 0) s_key[w] = mf > low ? gain_key(mf - 1u, (mt << lgC) | rank) : 0ull;
    }
    __syncthreads();  // every warp's key is in
    gain_t W = 0ull;
    int good = 1;
    if (a.C == 1 || w < 2) W = warp_max_key(lane < PUSH_WARPS ? s_key[lane] : 0ull);
    if (a.C > 1) {
      if (w == 0 && lane < a.C)
        st_async_u64(map_rank(smem_addr(&s_res[par][rank]), (uint32_t)lane), W,
                     map_rank(smem_addr(&s_bar[par]), (uint32_t)lane));
      if (w == 1 && W != 0ull) {  // this block's best row, likely a coming pick's
        const int t = key_token(W);
        if (t != pref && lane == 0) prefetch_l2(R + (size_t)t * a.ldc, (uint32_t)(4 * a.ldc));
        pref = t;
      }
      if (lane == 0 && !mbar_test(&s_bar[par], (uint32_t)((step - 1) >> 1) & 1u)) {
        const uint64_t t0 = globaltimer_ns();
        uint32_t spins = 0;
        while (!mbar_test(&s_bar[par], (uint32_t)((step - 1) >> 1) & 1u)) {
          if ((++spins & 15u) == 0) {
            if (ld_volatile_i32(a.status) != 0) { good = 0; break; }
            if (globaltimer_ns() - t0 > a.timeout_ns) {
              set_status(a.status, CP_ETIMEOUT);
              good = 0;
              break;
            }
          }
        }
      }
      good = __shfl_sync(0xFFFFFFFFu, good, 0);
      if (!good && lane == 0) s_fail = 1;
      W = good ? warp_max_key(lane < a.C ? *(volatile gain_t*)&s_res[par][lane] : 0ull) : 0ull;
    }
    const int pick = W ? key_token(W) : -1;
    if (pick < 0) {
      // no gain within the scale's reach: the rounds that follow fit it (or a
      // wait that ran out)
      if (lane == 0 && good) s_qn = -1;
    } else {
      if (rank == 0 && threadIdx.x == 0) {
        a.order32[(size_t)b * a.K + step] = pick;
        if (a.out_gains) a.out_gains[(size_t)b * a.K + step] = key_gain(W);
      }
      // ---- S <- S u {t*} (Eq. sgs_update): the targets whose m drops
      const float4* row = reinterpret_cast<const float4*>(R + (size_t)pick * a.ldc);
      const float4* m4 = reinterpret_cast<const float4*>(sm_m);
      const int nq = ncols >> 2;
      for (int i0 = w * 32; i0 < nq; i0 += 4 * PUSH_THREADS) {
        float4 c[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + u * PUSH_THREADS + lane;
          c[u] = i < nq ? __ldg(row + i) : make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (i0 + u * PUSH_THREADS >= nq) break;  // warp-uniform
          const int i = i0 + u * PUSH_THREADS + lane;
          const float4 mm = i < nq ? m4[i] : make_float4(0.f, 0.f, 0.f, 0.f);
          const uint32_t low = (c[u].x < mm.x ? 1u : 0u) | (c[u].y < mm.y ? 2u : 0u) |
                               (c[u].z < mm.z ? 4u : 0u) | (c[u].w < mm.w ? 8u : 0u);
          uint32_t bal[4];
          int n = 0;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            bal[e] = __ballot_sync(0xFFFFFFFFu, (low >> e) & 1u);
            n += __popc(bal[e]);
          }
          if (n != 0) {  // warp-uniform
            int at = 0;
            if (lane == 0) at = atomicAdd(&s_qn, n);
            at = __shfl_sync(0xFFFFFFFFu, at, 0);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              if ((low >> e) & 1u)
                queue[at + __popc(bal[e] & ((1u << lane) - 1u))] = (uint32_t)(4 * i + e);
              at += __popc(bal[e]);
            }
          }
        }
      }
    }
    __syncthreads();  // the lowered targets are listed
    if (s_fail != 0 || s_qn < 0) {  // block-uniform; this step is not taken
      ok = s_fail == 0;
      break;
    }
    last = pick;
    // ---- LW lanes per lowered target: its live candidates lose what the drop
    // took; the entries that stay live are packed to the list's front.  Four
    // entries a lane are in flight, and the next target's length and costs
    // load meanwhile.
    constexpr int PER = 32 / LW;  // targets a warp takes at a time
    const int qn = s_qn, sub = lane / LW, gl = lane & (LW - 1);
    int j = 0, len = 0;
    float mn = 0.0f, vj = 0.0f;
    auto next = [&](int q) {
      len = 0;
      if (q < qn) {
        j = (int)queue[q];
        len = (int)__ldcg(a.lens + ((size_t)bl * N + j) * a.C + rank);
        mn = __ldg(R + (size_t)pick * a.ldc + j);
        vj = __ldg(v + j);
      }
    };
    next(PER * w + sub);
#pragma unroll 1
    for (int q = PER * w; q < qn; q += PER * PUSH_WARPS) {
      const int jc = j, lenc = len;
      const float mnc = mn, mo = sm_m[j], vc = vj;
      const size_t lj = ((size_t)bl * N + jc) * a.C + rank;
      Entry* L = a.lists + lj * a.NC;
      const bool on = q + sub < qn;
      next(q + PER * PUSH_WARPS + sub);
      int out = 0;
#pragma unroll 1
      for (int i0 = gl; __any_sync(0xFFFFFFFFu, i0 - gl < lenc); i0 += 4 * LW) {
        Entry x[4];
        gain_t d[4];
        uint32_t old[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          x[u] = i0 + LW * u < lenc ? __ldcg(L + i0 + LW * u) : make_uint2(0u, 0x7F800000u);
#pragma unroll
        for (int u = 0; u < 4; ++u)
          d[u] = chunk_low(g_lo, x[u].x, vc, mo, mnc, __uint_as_float(x[u].y), fx, old[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          chunk_high(g_hi, x[u].x, d[u], old[u]);
          if (d[u] != 0ull) s_dirty[x[u].x >> a.lgS] = 1u;
          const bool stay = __uint_as_float(x[u].y) < mnc;
          uint32_t mask = __ballot_sync(0xFFFFFFFFu, stay);
          if (LW < 32) mask = (mask >> (lane & (32 - LW))) & ((1u << (LW & 31)) - 1u);
          const int p = out + __popc(mask & ((1u << gl) - 1u));
          if (stay && p != i0 + LW * u) __stcg(L + p, x[u]);
          out += __popc(mask);
        }
      }
      if (gl == 0 && on) {
        my_ent += (uint32_t)lenc;
        if (out != lenc) __stcg(a.lens + lj, (uint32_t)out);
        sm_m[jc] = mnc;
      }
    }
    mean8 += qn - (mean8 >> 3);
    __syncthreads();  // gains and m are settled
    if (threadIdx.x == 0) s_qn = 0;
  }

  unsigned long long* cstats = reinterpret_cast<unsigned long long*>(
      reinterpret_cast<unsigned char*>(a.status) + kCallStatsOffset);
  if ((lane & (LW - 1)) == 0 && my_ent) {
    atomicAdd(&cstats[0], (unsigned long long)my_ent);
    atomicAdd(&cstats[2], 8ull * (unsigned long long)my_ent);
  }
  if (rank == 0 && threadIdx.x == 0) {
    atomicAdd(&cstats[1], (unsigned long long)step);
    atomicAdd(&cstats[2], 4ull * (unsigned long long)step * (unsigned long long)ncols);
  }
  // the state for the rounds that follow
  if (ok && rank == (last & (a.C - 1)) && threadIdx.x == 0) g_hi[last >> lgC] = 0xFFFFFFFFu;
  __syncthreads();
  for (int tl = threadIdx.x; tl < nown; tl += PUSH_THREADS)
    a.gains[(size_t)b * N + ((tl << lgC) | rank)] = ((gain_t)g_hi[tl] << 32) | g_lo[tl];
  if (rank == 0) {
    for (int j = threadIdx.x; j < N; j += PUSH_THREADS) a.m_out[(size_t)bl * N + j] = sm_m[j];
    if (threadIdx.x == 0) a.stop[bl] = ok ? step : a.K;
  }
  if (!ok) {  // a peer's last key may still be on its way here: let it land
    const uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 500000ull) {
    }
  }
  hw_cluster_sync();  // nobody leaves while a peer may still write to its shared memory
}

// ---------------------------------------------------------------------------
// The lists of a dense scene for the rounds below, a warp per target: the C
// parts of its list copied into one, side by side with the other targets'
// (the parts lie 8 N bytes a target apart, a page or more each), and every
// candidate's row of live targets (room for row_room(N) entries; a longer row
// only counts).  A list that finds no room in the joined region is joined where
// it is: parts move toward the list's front, each chunk read before it is
// written.
// ---------------------------------------------------------------------------
constexpr int RD_ROW = 512;
__host__ __device__ constexpr int row_room(int64_t N) { return N < RD_ROW ? (int)N : RD_ROW; }

__global__ void __launch_bounds__(256) k_join_lists(Entry* __restrict__ lists,
                                                    const uint32_t* __restrict__ lens, int N, int C,
                                                    int lgC, int NC, size_t join0, uint32_t room,
                                                    uint32_t* __restrict__ cursor,
                                                    uint2* __restrict__ span,
                                                    uint32_t* __restrict__ row_len,
                                                    Entry* __restrict__ rows) {
  const int j = blockIdx.x * 8 + (threadIdx.x >> 5), bl = blockIdx.y, lane = threadIdx.x & 31;
  if (j >= N) return;
  const size_t lj = ((size_t)bl * N + j) * C;
  const uint32_t mine = lane < C ? lens[lj + lane] : 0u;
  const uint32_t total = __reduce_add_sync(0xFFFFFFFFu, mine);
  uint32_t at = 0u;
  if (lane == 0 && total) at = atomicAdd(cursor + bl, total);
  at = __shfl_sync(0xFFFFFFFFu, at, 0);
  size_t to = lj * NC;
  if (at <= room && total <= room - at) to = join0 + (size_t)bl * room + at;
  uint32_t* rl = row_len + (size_t)bl * N;
  const uint32_t rr = (uint32_t)row_room(N);
  Entry* rw = rows + (size_t)bl * N * rr;
  int out = 0;
  for (int r = 0; r < C; ++r) {
    const int len = (int)__shfl_sync(0xFFFFFFFFu, mine, r);
    const Entry* S = lists + (lj + r) * NC;
    for (int i0 = 0; i0 < len; i0 += 32) {
      const int n = min(32, len - i0);
      Entry x = make_uint2(0u, 0u);
      if (lane < n) x = S[i0 + lane];
      __syncwarp();
      if (lane < n) {
        const uint32_t t = (x.x << lgC) | (uint32_t)r;
        lists[to + out + lane] = make_uint2(t, x.y);
        const uint32_t p = atomicAdd(rl + t, 1u);
        if (p < rr) rw[(size_t)t * rr + p] = make_uint2((uint32_t)j, x.y);
      }
      out += n;
    }
  }
  if (lane == 0) span[(size_t)bl * N + j] = make_uint2((uint32_t)to, (uint32_t)out);
}

// ---------------------------------------------------------------------------
// Many picks a round.  Among a set S of candidates with exact gains the
// greedy can run on S alone for as long as S's best gain stays above a bound
// on every gain outside S: gains only fall, so nothing outside S can win
// before that.  And a member of S whose gain is above those of all members
// it shares a live target with will be picked with the gain it has: none of
// them can come first.  So all such members are picked at once, their order
// in the selection being that of their gains.  A round
//  - takes the best candidates of 32 slices (t mod 32, so that neighbours in
//    space fall into different ones), up to RD_TOP of each, and the largest
//    gain left out as the bound;
//  - brings their live targets (a few dozen entries each) into shared memory;
//  - repeats: rank the members above the bound, find those that are first on
//    all their live targets (a table of least ranks by target; targets that
//    collide in it only hold a member back), pick them, lower m, update the
//    members' gains;
//  - puts its picks in the order of their gains, and updates the lists of all
//    targets it lowered at once, as single picks would have done one after
//    the other (terms add up without an order).
// Where more members than picks to make are above the bound, only those
// before the first one held back are picked, up to the number to make.
// One block per scene, no waits on other blocks.  A round is a chain of a
// few dozen barriers with a shared-memory or L2 latency or two between each
// pair, so what counts is the number of rounds: 1229 picks of 8192 take 187
// decisions, the single picks before them among these.
//
// A candidate whose row does not fit leaves S and raises the bound to its
// gain; when that leaves no pick (or the best gains agree in their 24 bits
// with one outside) the best candidate is picked alone, its row read in
// pieces from the cost (or the slab).
// ---------------------------------------------------------------------------
constexpr int RD_WARPS = 32, RD_THREADS = 32 * RD_WARPS;
constexpr int RD_EPT = 4;                        // row entries a thread holds at most
constexpr int RD_EMAX = RD_EPT * RD_THREADS;     // ... and a round
// Members a slice gives at most (fewer where the rows' room is small, see
// launch_rounds).  Selection, ms, at 2 / 4 / 8: N = 8192 3.51 / 3.26 / 4.00, 4
// local scenes of 6272 1.53 / 1.53 / 2.42: fewer picks a round on one side, more
// rows to stage and rank on the other.
constexpr int RD_TOP = 4;
constexpr int RD_MEMBERS = RD_TOP * RD_WARPS;
constexpr uint32_t NO_ENTRY = 0xFFFFFFFFu;
constexpr uint32_t NO_RANK = 0x7FFFFFFFu;

struct RoundArgs {
  const float* rows;       // dense: cost [B][N][ldc]; local: slab [B][N][g]
  const int32_t* nbr;      // local: [B][N][kk]
  const float* v;          // [B][N]
  const gain_t* gains0;    // [B][N] gains at the start (high word ~0: selected)
  const float* m_in;       // dense: [scenes of the wave][N] coverage cost at the start
  const int* start;        // dense: [scenes of the wave] first step to take
  Entry* lists;
  uint2* span;             // [scenes][N] (offset, length)
  uint32_t* row_len;       // dense: [scenes of the wave][N]
  Entry* row_ent;          // dense: [scenes of the wave][N][row_room(N)]
  int32_t* order32;        // [B][K]
  float* out_gains;        // [B][K] or null
  double* objective;       // [B] or null
  int* status;
  int64_t ldc;
  const int* fxs;          // [B] the scenes' scales, or null: fx
  size_t list_step;        // local: entries between the lists of adjacent scenes
  float m0;
  int fx;
  int N, K, g, kk;
  int S;                   // candidates a slice, ceil(N / 32) made odd
  int emax;                // row entries a round holds, at most RD_EMAX
  int top;                 // members a slice gives at most, at most RD_TOP
  int tmask;               // size of the table of least ranks - 1
  int scene0;
  uint32_t off_lo, off_hi, off_ent, off_em, off_qm, off_qj, off_bits, off_tab;  // dynamic shared memory
};

template <int W>
struct Lanes {
  static constexpr int value = W;
};
// Barrier of the first n warps.
__device__ __forceinline__ void warps_sync(int n) {
  asm volatile("bar.sync 1, %0;" ::"r"(32 * n) : "memory");
}

// How far a gain of this key, and so any smaller one, can be shifted up
// without reaching the sign.
__device__ __forceinline__ int gains_shift(gain_t key, int fx) {
  const uint32_t bits = (uint32_t)(key >> 32) - 1u;
  return bits ? min(31, fx - 2 - (int)(bits >> 23)) : 31;
}

// The gains (all 0 before) from the lists, a warp per target.
__device__ __noinline__ void sum_lists(const Entry* lists, const uint2* span, const float* v,
                                       const float* m, int N, int S, int fx, uint32_t* g_lo,
                                       uint32_t* g_hi) {
#pragma unroll 1
  for (int j = threadIdx.x >> 5; j < N; j += RD_WARPS) {
    const uint2 sp = __ldcg(span + j);
    const float vj = __ldg(v + j), mj = m[j];
#pragma unroll 1
    for (uint32_t i = threadIdx.x & 31; i < sp.y; i += 32) {
      const Entry x = __ldcg(lists + sp.x + i);
      const uint32_t at = (x.x & 31u) * (uint32_t)S + (x.x >> 5);
      const gain_t d = gain_term(vj, mj, __uint_as_float(x.y), fx);
      if (d == 0ull) continue;
      const uint32_t old = atomicAdd(g_lo + at, (uint32_t)d);
      const uint32_t dh = (uint32_t)(d >> 32) + (old > ~(uint32_t)d ? 1u : 0u);
      if (dh) atomicAdd(g_hi + at, dh);
    }
  }
}

template <bool LOCAL>
__global__ void __launch_bounds__(RD_THREADS, 1) k_sgs_rounds(const __grid_constant__ RoundArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  float* sm_m = reinterpret_cast<float*>(smem);                    // [N] coverage cost
  // gains as two words, slice after slice: candidate t at (t % 32) S + t / 32
  // (S odd: candidates with adjacent indices, often on one list, fall into
  // different banks)
  uint32_t* g_lo = reinterpret_cast<uint32_t*>(smem + a.off_lo);   // [32 S]
  uint32_t* g_hi = reinterpret_cast<uint32_t*>(smem + a.off_hi);   // [32 S]
  Entry* ent = reinterpret_cast<Entry*>(smem + a.off_ent);         // [emax] (member << 16 | j, cost)
  float* ent_m = reinterpret_cast<float*>(smem + a.off_em);        // [emax] their targets' m
  float* q_m = reinterpret_cast<float*>(smem + a.off_qm);          // [emax] lowered targets: old m
  uint16_t* q_j = reinterpret_cast<uint16_t*>(smem + a.off_qj);    // [emax] ... and index
  uint32_t* bits = reinterpret_cast<uint32_t*>(smem + a.off_bits);  // [ceil(N / 32)] lowered this round
  uint32_t* tab = reinterpret_cast<uint32_t*>(smem + a.off_tab);    // [tmask + 1] least rank by target
  __shared__ int s_top[RD_TOP][RD_WARPS];    // a slice's best candidates
  __shared__ int s_left[RD_WARPS];           // bound on a slice's other gains, high word (-1: none)
  __shared__ uint32_t s_mlo[RD_MEMBERS], s_mhi[RD_MEMBERS];  // members' gains
  __shared__ int s_mtok[RD_MEMBERS];         // members (-1: not in S, or picked)
  __shared__ gain_t s_mkey[RD_MEMBERS];      // their keys (0: none, or not above the bound)
  __shared__ int s_rank[RD_MEMBERS];
  __shared__ uint32_t s_held[RD_MEMBERS];    // shares a live target with a better member
  __shared__ int s_pick[RD_MEMBERS];
  __shared__ gain_t s_pkey[RD_MEMBERS];      // the picks' keys
  __shared__ gain_t s_best[RD_WARPS];
  __shared__ gain_t s_tau;                   // one more than the largest gain outside S can be (0: none)
  __shared__ int s_fx;                       // the gains' scale (sgs_gain.cuh)
  __shared__ int s_sh;                       // every gain left is below 2^(63 - sh)
  __shared__ int s_nm, s_ne, s_qn, s_np, s_cut, s_nv[2];

  const int bl = blockIdx.x, b = a.scene0 + bl;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int N = a.N, S = a.S;
  const float* v = a.v + (size_t)b * N;
  const float* R = a.rows + (size_t)b * N * (LOCAL ? (size_t)a.g : (size_t)a.ldc);
  const int32_t* NB = LOCAL ? a.nbr + (size_t)b * N * a.kk : nullptr;
  uint2* span = a.span + (size_t)bl * N;
  Entry* lists = LOCAL ? a.lists + (size_t)bl * a.list_step : a.lists;
  uint32_t my_ent = 0u, my_row = 0u, my_rounds = 0u;  // at most N^2 < 2^32 each

  int step = LOCAL ? 0 : a.start[bl];
  for (int j = threadIdx.x; j < N; j += RD_THREADS)
    sm_m[j] = LOCAL ? a.m0 : a.m_in[(size_t)bl * N + j];
  for (int p = threadIdx.x; p < 32 * S; p += RD_THREADS) {
    const int t = ((p % S) << 5) | (p / S);
    const gain_t x = t < N ? a.gains0[(size_t)b * N + t] : ~0ull;
    g_lo[p] = (uint32_t)x;
    g_hi[p] = (uint32_t)(x >> 32);
  }
  for (int i = threadIdx.x; i < (N + 31) / 32; i += RD_THREADS) bits[i] = 0u;
  for (int i = threadIdx.x; i <= a.tmask; i += RD_THREADS) tab[i] = NO_RANK;
  if (threadIdx.x == 0) {
    s_np = 0;
    s_fx = a.fxs ? a.fxs[b] : a.fx;
    s_sh = 0;
  }
  __syncthreads();

  while (step < a.K) {
    ++my_rounds;
#pragma unroll 1
    for (int i = lane; i < s_np; i += 32) {  // the last round's picks are no candidates any more
      const int t = s_pick[i];
      if ((t & 31) == w) g_hi[w * S + (t >> 5)] = 0xFFFFFFFFu;
    }
    __syncwarp();
    // ---- the slice's best candidates, by the 31 bits of their gains that
    // start at the last picks' leading one (no gain left is above those) with
    // the place in the lane's run in the low 5 (negative: selected, or none):
    // each lane its three best, then the warp's best of those heads in turn;
    // a lane whose three are used up bounds its rest by the third.  Fixed bits
    // of the scale, ranked by before, did not tell late gains apart: rounds of
    // a selection and ms, then / now, 4096 of 16384 tokens 972 / 534 and 29.3 /
    // 15.0 (with as many members a slice); 1229 of 8192 at m0 = 1000 1002 / 199
    // and 12.4 / 4.0; at the default m0 190 / 189 and 3.24 / 3.27 (the shift and
    // the variable scale)
    int cnt = 0, left = -1;
    const int sh = s_sh;
    {
      int v1 = -1, v2 = -1, v3 = -1;
#pragma unroll 4
      for (int i = lane, q = 0; i < S; i += 32, ++q) {
        const uint32_t top = __funnelshift_l(g_lo[w * S + i], g_hi[w * S + i], sh);
        const int x = (int)((top & 0xFFFFFFE0u) | (uint32_t)q);
        v3 = max(v3, min(v2, x));
        v2 = max(v2, min(v1, x));
        v1 = max(v1, x);
      }
      const int third = v3;
      bool real = true;  // the head is a candidate, not a bound
#pragma unroll 1
      for (; cnt < a.top; ++cnt) {
        const int best = __reduce_max_sync(0xFFFFFFFFu, v1);
        const uint32_t who = __ballot_sync(0xFFFFFFFFu, v1 == best && real);
        if (best < 0 || who == 0u) break;  // warp-uniform
        if (lane == __ffs(who) - 1) {
          s_top[cnt][w] = (((best & 31) * 32 + lane) << 5) | w;
          v1 = v2;
          v2 = v3;
          v3 = -1;
          if (v1 < 0) {
            v1 = third;
            real = false;
          }
        }
      }
      left = __reduce_max_sync(0xFFFFFFFFu, v1);
      if (left >= 0) left |= 31;
      if (lane == 0) s_left[w] = left;
    }
    if (threadIdx.x == 0) {
      s_nm = 0;
      s_ne = 0;
      s_qn = 0;
      s_nv[0] = s_nv[1] = 0;
      s_tau = 0ull;
    }
    __syncthreads();  // every slice's bound is in
    // ---- S: the slices' candidates above the leading bits of all left out
    left = __reduce_max_sync(0xFFFFFFFFu, s_left[lane]);
    if (threadIdx.x == 0) {
      s_np = 0;
      if (left >= 0) atomicMax(&s_tau, (gain_t)((uint32_t)left + 1u) << (32 - sh));
    }
    if (cnt > 0) {
      const int t = lane < cnt ? s_top[lane][w] : 0;
      const uint32_t lo = lane < cnt ? g_lo[w * S + (t >> 5)] : 0u;
      const uint32_t hi = lane < cnt ? g_hi[w * S + (t >> 5)] : 0u;
      const uint32_t in = __ballot_sync(
          0xFFFFFFFFu, lane < cnt && (int)__funnelshift_l(lo, hi, sh) > left);
      if (in) {
        int i = 0;
        if (lane == 0) i = atomicAdd(&s_nm, __popc(in));
        i = __shfl_sync(0xFFFFFFFFu, i, 0) + lane;
        if ((in >> lane) & 1u) {  // in order, so lanes 0 .. popc - 1
          s_mtok[i] = t;
          s_mlo[i] = lo;
          s_mhi[i] = hi;
        }
      }
    }
    __syncthreads();
    // ---- the members' live targets (packed to the row's front on the dense
    // path): rows of up to 64 entries are held in registers between the count
    // and the write, longer ones are read twice
    const int nm = s_nm, rr = row_room(N);
#pragma unroll 1
    for (int i = w; i < nm; i += RD_WARPS) {
      const int t = s_mtok[i];
      Entry* rw = LOCAL ? nullptr : a.row_ent + ((size_t)bl * N + t) * rr;
      // entry q of the row of n, dead past it
      auto fetch = [&](int q, int n) -> Entry {
        Entry e = make_uint2(0u, 0x7F800000u);
        if (q < n) {
          if (LOCAL) {
            e.x = q == 0 ? (uint32_t)t : (uint32_t)__ldg(NB + (size_t)t * a.kk + q - 1);
            e.y = __float_as_uint(__ldg(R + (size_t)t * a.g + q));
          } else {
            e = __ldcg(rw + q);
          }
        }
        return e;
      };
      Entry x[2];
      x[0] = fetch(lane, LOCAL ? a.g : rr);
      x[1] = fetch(32 + lane, LOCAL ? a.g : rr);
      const int len = LOCAL ? a.g : (int)__ldcg(a.row_len + (size_t)bl * N + t);
      const bool stored = LOCAL || len <= rr;  // a longer row is not kept
      const uint32_t lt = (1u << lane) - 1u;
      uint32_t mask[2];
      float m[2];
      int n = 0, n2;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int q = 32 * u + lane;
        const bool in = stored && q < len;
        m[u] = sm_m[in ? x[u].x : 0u];
        mask[u] = __ballot_sync(0xFFFFFFFFu, in && __uint_as_float(x[u].y) < m[u]);
        const int p = n + __popc(mask[u] & lt);
        if (!LOCAL && ((mask[u] >> lane) & 1u) && p != q) __stcg(rw + p, x[u]);
        n += __popc(mask[u]);
      }
      n2 = n;
      if (stored)
#pragma unroll 1
        for (int k0 = 64; k0 < len; k0 += 64) {
          Entry y[2];
          y[0] = fetch(k0 + lane, len);
          y[1] = fetch(k0 + 32 + lane, len);
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int q = k0 + 32 * u + lane;
            const bool live = __uint_as_float(y[u].y) < sm_m[y[u].x];
            const uint32_t mk = __ballot_sync(0xFFFFFFFFu, live);
            const int p = n2 + __popc(mk & lt);
            if (!LOCAL && live && p != q) __stcg(rw + p, y[u]);
            n2 += __popc(mk);
          }
        }
      int at = 0;
      if (lane == 0 && n2) at = atomicAdd(&s_ne, n2);
      at = __shfl_sync(0xFFFFFFFFu, at, 0);
      const bool fits = stored && at + n2 <= a.emax;
      // the last places are filled even when the row does not fit
      auto put = [&](const Entry& e, float mj, bool live, uint32_t mk) {
        const int p = at + __popc(mk & lt);
        if (live && p < a.emax) {
          ent[p] = make_uint2(fits ? ((uint32_t)i << 16) | e.x : NO_ENTRY, e.y);
          ent_m[p] = mj;
        }
        at += __popc(mk);
      };
#pragma unroll
      for (int u = 0; u < 2; ++u) put(x[u], m[u], (mask[u] >> lane) & 1u, mask[u]);
      if (n2 > n) {
        __syncwarp();  // the packed row is visible to the whole warp
        const int rn = LOCAL ? len : n2;
#pragma unroll 1
        for (int q = (LOCAL ? 64 : n) + lane; q - lane < rn; q += 32) {
          const Entry e = fetch(q, rn);
          const float mj = sm_m[e.x];
          const bool live = __uint_as_float(e.y) < mj;
          put(e, mj, live, __ballot_sync(0xFFFFFFFFu, live));
        }
      }
      if (lane == 0) {
        my_row += stored ? (uint32_t)len : 0u;
        if (!LOCAL && stored && n2 != len) __stcg(a.row_len + (size_t)bl * N + t, (uint32_t)n2);
        if (!fits) {
          s_mtok[i] = -1;
          atomicMax(&s_tau, (((gain_t)s_mhi[i] << 32) | s_mlo[i]) + 1ull);
        }
      }
    }
    __syncthreads();
    // ---- picks from S while its best stays above what is outside, by the
    // first nw warps
    const int ne = min(s_ne, a.emax);
    const int nw = min(RD_WARPS, max(4, (ne + 31) / 32)), nt = 32 * nw;
    if (w < nw) {
      const int fx = s_fx;
      // a thread's entries
      float ec[RD_EPT], em[RD_EPT];
      uint32_t ej[RD_EPT];
#pragma unroll
      for (int u = 0; u < RD_EPT; ++u) {
        const int e = threadIdx.x + u * nt;
        const Entry x = e < ne ? ent[e] : make_uint2(NO_ENTRY, 0u);
        const bool on = x.x != NO_ENTRY;
        ej[u] = on ? x.x : 0u;
        ec[u] = on ? __uint_as_float(x.y) : INFINITY;
        em[u] = on ? ent_m[e] : -INFINITY;  // m never falls below that
      }
      // 24 bits of the largest gain outside S, + 1 (0: none), or those from
      // which on the scale fits
      const uint32_t out = max(s_tau ? gain_bits(s_tau - 1ull, fx) + 1u : 0u, gain_floor(fx));
      const int mi = threadIdx.x;  // a thread's member (nt >= RD_MEMBERS)
      for (int it = 0;; ++it) {
        // the members' keys, of those whose 24 bits are above the bound
        if (mi < RD_MEMBERS) {
          gain_t key = 0ull;
          const int t = mi < nm ? s_mtok[mi] : -1;
          if (t >= 0) {
            const uint32_t f = gain_bits(((gain_t)s_mhi[mi] << 32) | s_mlo[mi], fx) + 1u;
            if (f > out) key = gain_key(f - 1u, t);
          }
          s_mkey[mi] = key;
          s_held[mi] = 0u;
          const int n = __popc(__ballot_sync(0xFFFFFFFFu, key != 0ull));
          if (lane == 0 && n) atomicAdd(&s_nv[it & 1], n);
          if (mi == 0) {
            s_cut = RD_MEMBERS;
            s_nv[(it + 1) & 1] = 0;
          }
        }
        warps_sync(nw);
        const int nv = s_nv[it & 1], room = a.K - step - s_np;
        if (nv == 0 || room == 0) break;  // the same in every warp
        // their ranks, four lanes a member
        for (int i0 = 0; i0 < nm; i0 += nt / 4) {
          const int i = i0 + (int)(threadIdx.x >> 2);
          const gain_t mine = i < nm ? s_mkey[i] : 0ull;
          int r = 0;
#pragma unroll 4
          for (int o = lane & 3; o < nm; o += 4) r += s_mkey[o] > mine ? 1 : 0;
          r += __shfl_xor_sync(0xFFFFFFFFu, r, 1);
          r += __shfl_xor_sync(0xFFFFFFFFu, r, 2);
          if ((lane & 3) == 0 && i < nm) s_rank[i] = mine ? r : (int)NO_RANK;
        }
        warps_sync(nw);
        // the least rank on each target ...
        int er[RD_EPT];
#pragma unroll
        for (int u = 0; u < RD_EPT; ++u) {
          er[u] = (int)NO_RANK;
          if (u * nt < ne && ec[u] < em[u]) er[u] = s_rank[ej[u] >> 16];
          if (er[u] != (int)NO_RANK) atomicMin(tab + (ej[u] & (uint32_t)a.tmask), (uint32_t)er[u]);
        }
        warps_sync(nw);
        // ... holds back the members that are not it
#pragma unroll
        for (int u = 0; u < RD_EPT; ++u) {
          if (er[u] != (int)NO_RANK && tab[ej[u] & (uint32_t)a.tmask] < (uint32_t)er[u]) {
            s_held[ej[u] >> 16] = 1u;
            if (nv > room) atomicMin(&s_cut, er[u]);
          }
        }
        warps_sync(nw);
        // S <- S u {t*} (Eq. sgs_update) for the others: their live entries,
        // one a target, lower m
        const int lim = nv > room ? min(s_cut, room) : RD_MEMBERS;
#pragma unroll
        for (int u = 0; u < RD_EPT; ++u) {
          if (er[u] != (int)NO_RANK) {
            tab[ej[u] & (uint32_t)a.tmask] = NO_RANK;
            if (er[u] < lim && s_held[ej[u] >> 16] == 0u) {
              const int j = (int)(ej[u] & 0xFFFFu);
              sm_m[j] = ec[u];
              const uint32_t bit = 1u << (j & 31);
              if (!(atomicOr(bits + (j >> 5), bit) & bit)) {
                const int q = atomicAdd(&s_qn, 1);
                q_j[q] = (uint16_t)j;
                q_m[q] = em[u];
              }
            }
          }
        }
        if (mi < nm && s_rank[mi] < lim && s_held[mi] == 0u) {
          const int p = atomicAdd(&s_np, 1);
          s_pick[p] = s_mtok[mi];
          s_pkey[p] = s_mkey[mi];
          s_mtok[mi] = -1;
        }
        warps_sync(nw);
        // a lowered target takes off the members that still covered it
#pragma unroll
        for (int u = 0; u < RD_EPT; ++u) {
          const float mj = u * nt < ne ? sm_m[ej[u] & 0xFFFFu] : INFINITY;
          if (mj < em[u]) {
            const uint32_t i = ej[u] >> 16;
            uint32_t old;
            const gain_t d = chunk_low(s_mlo, i, __ldg(v + (ej[u] & 0xFFFFu)), em[u], mj, ec[u], fx,
                                       old);
            chunk_high(s_mhi, i, d, old);
            em[u] = mj;
          }
        }
        warps_sync(nw);
      }
      // the picks in order, four lanes each
      const int np = s_np;
      for (int i0 = 0; i0 < np; i0 += nt / 4) {
        const int i = i0 + (int)(threadIdx.x >> 2);
        const gain_t mine = i < np ? s_pkey[i] : 0ull;
        int r = 0;
#pragma unroll 4
        for (int o = lane & 3; o < np; o += 4) r += s_pkey[o] > mine ? 1 : 0;
        r += __shfl_xor_sync(0xFFFFFFFFu, r, 1);
        r += __shfl_xor_sync(0xFFFFFFFFu, r, 2);
        if ((lane & 3) == 0 && i < np) {
          a.order32[(size_t)b * a.K + step + r] = s_pick[i];
          if (r == np - 1) s_sh = gains_shift(mine, fx);
          if (a.out_gains) a.out_gains[(size_t)b * a.K + step + r] = key_gain(mine);
        }
      }
    }
    __syncthreads();
    const int np = s_np;
    int pick = -1, len = 0;
    if (np == 0) {
      // ---- no pick from S: the best candidate alone, by its exact key
      const int fx = s_fx;
      gain_t best = 0ull;
#pragma unroll 1
      for (int i = lane; i < S; i += 32) {
        const uint32_t hi = g_hi[w * S + i];
        if ((int)hi < 0) continue;
        const gain_t key =
            gain_key(gain_bits(((gain_t)hi << 32) | g_lo[w * S + i], fx), (i << 5) | w);
        best = key > best ? key : best;
      }
      best = warp_max_key(best);
      if (lane == 0) s_best[w] = best;
      __syncthreads();
      best = warp_max_key(s_best[lane]);
      pick = best ? key_token(best) : -1;
      if (pick < 0) {  // never expected: no candidate left (block-uniform)
        if (threadIdx.x == 0 && atomicCAS(a.status, 0, CP_EDEVICE) == 0) {
          a.status[4] = step;
          a.status[5] = b;
          a.status[6] = 0;
          a.status[7] = pick;
        }
        return;
      }
      if ((uint32_t)(best >> 32) <= gain_floor(fx)) {  // block-uniform
        // ---- the scale no longer fits: the gains afresh at one that does,
        // a warp per target's list
        const int fit = gain_refit((uint32_t)(best >> 32) - 1u, fx, 32 - __clz(N));
        for (int p = threadIdx.x; p < 32 * S; p += RD_THREADS)
          if ((int)g_hi[p] >= 0) g_lo[p] = g_hi[p] = 0u;
        __syncthreads();
        if (threadIdx.x == 0) {
          s_fx = fit;
          s_sh = 0;
        }
        sum_lists(lists, span, v, sm_m, N, S, fit, g_lo, g_hi);
        __syncthreads();
        continue;
      }
      len = LOCAL ? a.g : N;
      if (threadIdx.x == 0) {
        s_sh = gains_shift(best, fx);
        a.order32[(size_t)b * a.K + step] = pick;
        if (a.out_gains) a.out_gains[(size_t)b * a.K + step] = key_gain(best);
        s_pick[0] = pick;
        s_np = 1;
        my_row += (uint32_t)len;
      }
    }
    // ---- the lists of the lowered targets; a lone pick's row in pieces
    int k0 = 0;
#pragma unroll 1
    do {
      if (pick >= 0) {
        if (threadIdx.x == 0) s_qn = 0;
        __syncthreads();
#pragma unroll 1
        for (int q = k0 + threadIdx.x; q < min(len, k0 + a.emax); q += RD_THREADS) {
          const int j = LOCAL ? (q == 0 ? pick : __ldg(NB + (size_t)pick * a.kk + q - 1)) : q;
          const float c = __ldg(R + (size_t)pick * (LOCAL ? (size_t)a.g : (size_t)a.ldc) + q);
          const float mj = sm_m[j];
          if (c < mj) {
            const int at = atomicAdd(&s_qn, 1);
            q_j[at] = (uint16_t)j;
            q_m[at] = mj;
            sm_m[j] = c;
          }
        }
        __syncthreads();
        k0 += a.emax;
      }
      // every live candidate of target q_j loses what the drop from q_m to m
      // took; the entries that stay live are packed to the list's front.  A
      // turn of this loop is a chain of latencies: 8 lanes take a list, 128
      // lists a turn of the block, while lists are short (4 to 30 entries for
      // most of a selection), 16 while they are long
      const int qn = s_qn;
      const int fx = s_fx;
      auto push = [&](auto width) {
        constexpr int W = decltype(width)::value;   // lanes a list
        constexpr int U = W == 16 ? 4 : 2;          // entries a lane has in flight
        const int gl = lane & (W - 1), gs = lane & (32 - W);
        constexpr uint32_t gm = (1u << W) - 1u;
#pragma unroll 1
        for (int q0 = (32 / W) * w; q0 < qn; q0 += RD_THREADS / W) {
          const int q = q0 + lane / W;
          const bool on = q < qn;
          const int j = (int)q_j[on ? q : q0];
          const uint2 sp = __ldcg(span + j);
          const float vj = __ldg(v + j);
          const float mo = q_m[on ? q : q0], mn = sm_m[j];
          if (on && gl == 0) bits[j >> 5] = 0u;
          Entry* L = lists + sp.x;
          const int n = on ? (int)sp.y : 0;
          int out = 0;
#pragma unroll 1
          for (int i0 = gl; __any_sync(0xFFFFFFFFu, i0 - gl < n); i0 += U * W) {
            Entry x[U];
            gain_t d[U];
            uint32_t old[U], at[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
              x[u] = i0 + W * u < n ? __ldcg(L + i0 + W * u) : make_uint2(0u, 0x7F800000u);
#pragma unroll
            for (int u = 0; u < U; ++u) {
              at[u] = (x[u].x & 31u) * (uint32_t)S + (x[u].x >> 5);
              d[u] = chunk_low(g_lo, at[u], vj, mo, mn, __uint_as_float(x[u].y), fx, old[u]);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
              chunk_high(g_hi, at[u], d[u], old[u]);
              const bool stay = __uint_as_float(x[u].y) < mn;
              const uint32_t mask = (__ballot_sync(0xFFFFFFFFu, stay) >> gs) & gm;
              const int p = out + __popc(mask & ((1u << gl) - 1u));
              if (stay && p != i0 + W * u) __stcg(L + p, x[u]);
              out += __popc(mask);
            }
          }
          if (gl == 0 && n) {
            my_ent += (uint32_t)n;
            if (out != n) __stcg(&span[j].y, (uint32_t)out);
          }
        }
      };
      if (pick >= 0 || s_ne > 24 * s_nm)
        push(Lanes<16>{});
      else
        push(Lanes<8>{});
      __syncthreads();  // gains are settled
    } while (k0 < len);
    step += max(np, 1);
  }

  unsigned long long* cstats = reinterpret_cast<unsigned long long*>(
      reinterpret_cast<unsigned char*>(a.status) + kCallStatsOffset);
  if ((lane & 7) == 0) {
    if (my_ent) atomicAdd(&cstats[0], (unsigned long long)my_ent);
    atomicAdd(&cstats[2], 8ull * ((unsigned long long)my_ent + my_row));
  }
  if (threadIdx.x == 0) atomicAdd(&cstats[1], (unsigned long long)my_rounds);
  if (a.objective) {
    const double F = objective_sum(sm_m, v, N);
    if (threadIdx.x == 0) a.objective[b] = F;
  }
}

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

// Scenes whose lists are held at once.  A dense scene's lists take 8 N^2
// bytes at their largest (twice its cost), its joined lists and rows up to
// 16 RD_ROW N more, so a large batch runs in waves: as many scenes as fit 24
// GB (entries are then numbered in 32 bits), whatever the batch, so that no
// larger batch needs less; at least one.
int64_t push_wave(int64_t B, int64_t N) {
  const double per = 8.0 * (double)N * (double)(N + PUSH_CMAX + 2 * row_room(N));
  const int64_t w = 24.0e9 > per ? (int64_t)(24.0e9 / per) : 1;
  return w < B ? w : B;
}

struct PushPlan {
  size_t gains, first, max_bits, zero_bytes, sums, first_bytes, fxs, lens, span, lists, m, stop, row_len,
      row_ent, total;
  size_t join0;  // dense: entries before the joined lists
  int64_t wave;
};
// wave > 0: that many scenes' dense lists at once.
PushPlan push_plan(int64_t B, int64_t N, int64_t g, int64_t wave) {
  PushPlan p{};
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t at = off;
    off = up256(off + (bytes > 0 ? bytes : 1));
    return at;
  };
  const size_t BN = (size_t)B * (size_t)N;
  p.gains = take(sizeof(gain_t) * BN);
  if (g < N) {
    p.wave = B;
    p.span = take(sizeof(uint2) * BN);
    p.lists = take(sizeof(Entry) * BN * (size_t)g);
  } else {
    p.first = take(sizeof(gain_t) * (size_t)B);
    p.max_bits = take(sizeof(uint32_t) * (size_t)B);
    p.zero_bytes = off;
    p.sums = take(sizeof(float) * BN);
    p.first_bytes = off;
    p.fxs = take(sizeof(int) * (size_t)B);
    p.wave = wave > 0 ? wave : push_wave(B, N);
    const size_t WN = (size_t)p.wave * (size_t)N;
    p.lens = take(sizeof(uint32_t) * WN * PUSH_CMAX);
    p.join0 = WN * (size_t)(N + PUSH_CMAX);
    p.lists = take(sizeof(Entry) * (p.join0 + WN * (size_t)row_room(N)));
    p.span = take(sizeof(uint2) * WN);
    p.m = take(sizeof(float) * WN);
    p.stop = take(sizeof(int) * (size_t)p.wave);
    p.row_len = take(sizeof(uint32_t) * (WN + (size_t)p.wave));  // and the joined lists' cursors
    p.row_ent = take(sizeof(Entry) * WN * (size_t)row_room(N));
  }
  p.total = off;
  return p;
}

int lg2(int x) {
  int l = 0;
  while ((1 << l) < x) ++l;
  return l;
}

// Shared-memory layout and derived sizes for clusters of C blocks.
size_t push_shape(PushArgs& a, int C, int64_t ncols) {
  a.C = C;
  a.lgC = lg2(C);
  a.NC = (int)((a.N + C - 1) / C);
  const int per = (a.NC + PUSH_WARPS - 1) / PUSH_WARPS;
  a.lgS = lg2(per < 32 ? 32 : per);
  a.off_q = (uint32_t)(sizeof(float) * ncols);
  a.off_lo = a.off_q + (uint32_t)(sizeof(uint32_t) * (size_t)a.N);
  a.off_hi = a.off_lo + (uint32_t)(sizeof(uint32_t) * (size_t)a.NC);
  return a.off_hi + sizeof(uint32_t) * (size_t)a.NC;
}

// The largest cluster, C0 halved as often as needed, that the device can
// hold; its launch configuration in cfg (attr must outlive it).
template <typename Fn>
int push_config(Fn fn, PushArgs& a, int C0, int64_t scenes, const DeviceInfo& di, cudaStream_t s,
                cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr) {
  for (int C = C0; C >= 1; C >>= 1) {
    const size_t smem = push_shape(a, C, a.ldc);
    if (smem + 2048 > (size_t)di.max_smem_optin) continue;
    CP_TRY_STATUS(allow_smem((const void*)fn, smem, "launch_sgs_push: smem attribute"));
    *cfg = cudaLaunchConfig_t{};
    cfg->gridDim = dim3((unsigned)(scenes * C));
    cfg->blockDim = dim3(PUSH_THREADS);
    cfg->dynamicSmemBytes = smem;
    cfg->stream = s;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = (unsigned)C;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg->attrs = attr;
    cfg->numAttrs = 1;
    if (C > 8) {
      int clusters = 0;
      if (cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
              cudaSuccess ||
          cudaOccupancyMaxActiveClusters(&clusters, (const void*)fn, cfg) != cudaSuccess ||
          clusters < scenes) {
        (void)cudaGetLastError();
        continue;
      }
    }
    return CP_OK;
  }
  note_message("launch_sgs_push: no cluster shape fits");
  return CP_EUNSUPPORTED;
}

// The rounds' launch: one block per scene, the row entries a round holds as
// many as the shared memory beside m and the gains takes.
template <typename Fn>
int launch_rounds(Fn fn, RoundArgs& a, int64_t scenes, const DeviceInfo& di, cudaStream_t s) {
  const int N = a.N;
  a.S = ((N + 31) / 32) | 1;
  a.off_lo = (uint32_t)((sizeof(float) * (size_t)N + 15) & ~(size_t)15);
  a.off_hi = a.off_lo + 128u * (uint32_t)a.S;
  a.off_ent = a.off_hi + 128u * (uint32_t)a.S;
  size_t smem = 0;
  const int tab = N > 12288 ? 2048 : 4096;
  a.tmask = tab - 1;
  for (a.emax = RD_EMAX;; a.emax >>= 1) {
    a.off_em = a.off_ent + (uint32_t)(sizeof(Entry) * (size_t)a.emax);
    a.off_qm = a.off_em + (uint32_t)(sizeof(float) * (size_t)a.emax);
    a.off_qj = a.off_qm + (uint32_t)(sizeof(float) * (size_t)a.emax);
    a.off_bits = a.off_qj + (uint32_t)(sizeof(uint16_t) * (size_t)a.emax);
    a.off_tab = a.off_bits + (uint32_t)(sizeof(uint32_t) * (size_t)a.S);
    smem = a.off_tab + sizeof(uint32_t) * (size_t)tab;
    if (smem + 7168 <= (size_t)di.max_smem_optin) break;
    if (a.emax <= 256) return CP_EUNSUPPORTED;
  }
  // Members whose rows do not all fit hold one another up: each that is left out
  // bounds the picks by its gain.  Selection, ms, at 4 / 3 / 2 a slice: with 1024
  // row entries (15000 tokens) a tenth kept 7.69 / 7.52 / 7.67, a quarter 8.71 /
  // 8.65 / 9.14, local 4.34 / 3.62 / 3.13; with 512 (16384) 13.97 / 10.22 / 9.22,
  // 15.30 / 11.41 / 10.79, local 7.02 / 5.80 / 4.45; 2048 fit.
  a.top = a.emax >= 2048 ? RD_TOP : (a.emax >= 1024 && a.g >= N ? 3 : 2);
  CP_TRY_STATUS(allow_smem((const void*)fn, smem, "launch_sgs_push: rounds smem attribute"));
  fn<<<(unsigned)scenes, RD_THREADS, smem, s>>>(a);
  return launch_status("launch_sgs_push: rounds");
}

int launch_push(const float* cost, int64_t ldc, const float* slab, const int32_t* nbr,
                const float* v, const DevParams& P, int64_t B, int64_t N, int64_t K,
                int32_t* order32, float* gains, double* objective, int* status, cudaStream_t s,
                const float* g0, void* ws, int64_t wave) {
  DeviceInfo di;
  if (device_info(&di) != CP_OK) return CP_ECUDA;
  const bool local = P.g < N;
  const PushPlan pl = push_plan(B, N, P.g, wave);
  unsigned char* base = static_cast<unsigned char*>(ws);
  gain_t* gains64 = reinterpret_cast<gain_t*>(base + pl.gains);
  const int fx0 = gain_fx(P.m0);                    // uncovered targets cost m0,
  const int fx = local ? fx0 : gain_fx_covered(P);  // covered ones no more than the largest cost
  RoundArgs r{};
  r.rows = local ? slab : cost;
  r.nbr = nbr;
  r.v = v;
  r.gains0 = gains64;
  r.lists = reinterpret_cast<Entry*>(base + pl.lists);
  r.span = reinterpret_cast<uint2*>(base + pl.span);
  r.order32 = order32;
  r.out_gains = gains;
  r.objective = objective;
  r.status = status;
  r.ldc = ldc;
  r.m0 = P.m0;
  r.fx = fx;
  r.N = (int)N;
  r.K = (int)K;
  r.g = P.g;
  r.kk = P.kk;
  if (local) {
    const dim3 per_token((unsigned)((N + 7) / 8), (unsigned)B);
    CP_TRY_STATUS(cuda_status(cudaMemsetAsync(r.span, 0, sizeof(uint2) * (size_t)(B * N), s),
                              "launch_sgs_push: lists"));
    k_rev_count<<<per_token, 256, 0, s>>>(nbr, (int)N, P.g, P.kk, r.span);
    CP_TRY_STATUS(last_launch_status());
    k_rev_scan<<<(unsigned)B, 1024, 0, s>>>((int)N, r.span);
    CP_TRY_STATUS(last_launch_status());
    k_rev_fill<<<per_token, 256, 0, s>>>(slab, nbr, v, (int)N, P.g, P.kk, P.m0, fx0, r.span,
                                         r.lists, gains64);
    CP_TRY_STATUS(last_launch_status());
    r.list_step = (size_t)N * (size_t)P.g;
    return launch_rounds(k_sgs_rounds<true>, r, B, di, s);
  }
  const gain_t* first = nullptr;
  CP_TRY_STATUS(launch_first_pick(cost, ldc, v, P, B, N, s, g0, ws, &first));
  r.row_len = reinterpret_cast<uint32_t*>(base + pl.row_len);
  r.row_ent = reinterpret_cast<Entry*>(base + pl.row_ent);
  r.m_in = reinterpret_cast<float*>(base + pl.m);
  r.start = reinterpret_cast<int*>(base + pl.stop);
  PushArgs a{};
  a.cost = cost;
  a.v = v;
  a.gains = gains64;
  a.first = first;
  a.lists = r.lists;
  a.lens = reinterpret_cast<uint32_t*>(base + pl.lens);
  a.m_out = reinterpret_cast<float*>(base + pl.m);
  a.stop = reinterpret_cast<int*>(base + pl.stop);
  a.order32 = order32;
  a.out_gains = gains;
  a.status = status;
  a.ldc = ldc;
  a.timeout_ns = P.timeout_ns;
  a.m0 = P.m0;
  a.fx = fx;
  a.N = (int)N;
  a.K = (int)K;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  if (fx != fx0) {  // m0 is well above every cost
    int* fxs = reinterpret_cast<int*>(base + pl.fxs);
    k_first_scale<<<(unsigned)B, 256, 0, s>>>(cost, ldc, first, (int)N, P.m0, fx0, fx, fxs);
    CP_TRY_STATUS(last_launch_status());
    a.fxs = r.fxs = fxs;
  }
  auto lists_fn = a.fxs ? k_live_lists<true> : k_live_lists<false>;
  if (cuda_status(cudaFuncSetAttribute(lists_fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)LL_SMEM),
                  "launch_sgs_push: lists smem attribute") != CP_OK)
    return CP_ECUDA;
  for (int64_t b0 = 0; b0 < B; b0 += pl.wave) {
    const int64_t nb = B - b0 < pl.wave ? B - b0 : pl.wave;
    // as many blocks a scene as let the wave's scenes run at once, 64
    // candidates a block or more (the whole selection, us, with 32 / 64 / 128 /
    // 256 at least: one scene of 300 220 / 221 / 230 / 243, of 700 307 / 313 /
    // 328 / 362, of 1500 481 / 481 / 497 / 554, of 3000 875 / 876 / 876 / 972; 4 of
    // 300 251 / 249 / 255 / 264, of 1500 568 / 568 / 572 / 611)
    int C0 = PUSH_CMAX;
    while (C0 > 1 && ((int64_t)C0 * nb > di.sm_count || N / C0 < 64)) C0 >>= 1;
    if (C0 < 2 && N > 12288) C0 = 2;
    // lanes a list (its part in one block: N / C candidates at most): short
    // parts leave most of a warp idle, and a list is a chain of latencies;
    // many blocks with long parts are bound by the shared-memory atomics.
    // Selection, ms, at 8 / 16 / 32: one scene of 1024 (C = 8) 0.304 / 0.317 /
    // 0.354, of 8192 (16) 2.87 / 2.92 / 3.25, of 16384 (16) 11.3 / 11.2 / 11.7;
    // 8 of 8192 (16) 4.45 / 4.32 / 4.46, 16 (8) 7.15 / 7.05 / 7.40, 32 (4) 8.71
    // / 8.24 / 7.99; 32 of 2048 (4) 0.99 / 0.98 / 1.03.
    const int64_t part = N / C0;
    auto push_fn = a.fxs                          ? k_sgs_push<16, true>
                   : part >= 2048                 ? k_sgs_push<32>
                   : (nb == 1 && part <= 512) ? k_sgs_push<8>
                                                  : k_sgs_push<16>;
    CP_TRY_STATUS(push_config(push_fn, a, C0, nb, di, s, &cfg, attr));
    a.scene0 = (int)b0;
    lists_fn<<<dim3((unsigned)((N + LL_COLS - 1) / LL_COLS), (unsigned)a.C, (unsigned)nb),
               32 * LL_WARPS, LL_SMEM, s>>>(cost, ldc, v, first, (int)N, a.C, a.lgC, a.NC,
                                            (int)b0, P.m0, fx, a.fxs, gains64, a.lists, a.lens);
    CP_TRY_STATUS(launch_status("launch_sgs_push: lists"));
    const cudaError_t e = cudaLaunchKernelEx(&cfg, push_fn, a);
    note_launch();
    CP_TRY_STATUS(cuda_status(e, "launch_sgs_push: steps"));
    uint32_t* cursor = r.row_len + (size_t)nb * (size_t)N;
    CP_TRY_STATUS(cuda_status(
        cudaMemsetAsync(r.row_len, 0, sizeof(uint32_t) * ((size_t)nb * (size_t)N + (size_t)nb), s),
        "launch_sgs_push: rows"));
    k_join_lists<<<dim3((unsigned)((N + 7) / 8), (unsigned)nb), 256, 0, s>>>(
        a.lists, a.lens, (int)N, a.C, a.lgC, a.NC, pl.join0, (uint32_t)(N * row_room(N)), cursor,
        r.span, r.row_len, r.row_ent);
    CP_TRY_STATUS(last_launch_status());
    r.scene0 = (int)b0;
    CP_TRY_STATUS(launch_rounds(k_sgs_rounds<false>, r, nb, di, s));
  }
  return CP_OK;
}

}  // namespace

int launch_first_pick(const float* cost, int64_t ldc, const float* v, const DevParams& P, int64_t B,
                      int64_t N, cudaStream_t s, const float* g0, void* ws, const gain_t** first_out,
                      float** bound, gain_t** zeros) {
  const PushPlan pl = push_plan(B, N, N, 1);
  unsigned char* base = static_cast<unsigned char*>(ws);
  uint32_t* max_bits = reinterpret_cast<uint32_t*>(base + pl.max_bits);
  float* sums = g0 ? reinterpret_cast<float*>(base + pl.sums) : nullptr;
  gain_t* first = reinterpret_cast<gain_t*>(base + pl.first);
  *first_out = first;
  if (bound) *bound = reinterpret_cast<float*>(base + pl.sums);
  if (zeros) *zeros = reinterpret_cast<gain_t*>(base + pl.gains);
  if (bound && !g0)  // 0x7E7E7E7E: 8e37
    CP_TRY_STATUS(cuda_status(cudaMemsetAsync(*bound, 0x7E, sizeof(float) * (size_t)(B * N), s),
                              "launch_first_pick: bounds"));
  CP_TRY_STATUS(cuda_status(cudaMemsetAsync(base + pl.gains, 0, pl.zero_bytes, s),
                            "launch_first_pick: gains"));
  if (g0) {
    k_first_bounds<<<dim3((unsigned)((N + 255) / 256), (unsigned)B), 256, 0, s>>>(
        g0, fst_apply_slots(ldc), (int)N, sums, max_bits);
    CP_TRY_STATUS(last_launch_status());
  }
  const int64_t groups = g0 ? (N + 255) / 256 : (N + 7) / 8;
  k_first_pick<<<dim3((unsigned)(groups < 512 ? groups : 512), (unsigned)B), 256, 0, s>>>(
      cost, ldc, v, (int)N, P.m0, gain_fx(P.m0), sums, max_bits, first);
  return last_launch_status();
}

size_t sgs_push_first_bytes(int64_t B, int64_t N) { return push_plan(B, N, N, 1).first_bytes; }
int64_t sgs_push_wave(int64_t B, int64_t N) { return push_wave(B, N); }

// A local selection's own lists; where the dense ones are small (64 MB) room
// for those, so that a program may try both on one workspace.
size_t sgs_push_ws_bytes(int64_t B, int64_t N, int64_t g, int64_t wave) {
  if (wave > 0) return push_plan(B, N, g, wave).total;
  const size_t dense = push_plan(B, N, N, 0).total;
  if (g >= N) return dense;
  const size_t local = push_plan(B, N, g, 0).total, small = (size_t)64 << 20;
  const size_t either = dense < small ? dense : small;
  return local > either ? local : either;
}

int launch_sgs_push(const float* cost, int64_t ldc, const float* slab, const int32_t* nbr,
                    const float* v, const DevParams& P, int64_t B, int64_t N, int64_t K,
                    int32_t* order32, float* gains, double* objective, int* status,
                    cudaStream_t s, const float* g0, void* ws, int64_t wave) {
  return launch_push(cost, ldc, slab, nbr, v, P, B, N, K, order32, gains, objective, status, s, g0,
                     ws, wave);
}

}  // namespace cp
