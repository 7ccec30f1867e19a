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
// in M_g(t) (k_rev_lists).
//
// What bounds a step is its chain of dependent latencies -- argmax, the
// winner's row, the changed targets' lists, the gain updates -- with block
// barriers between; nothing in it needs more than one SM except the first
// steps' long lists.  A scene therefore runs on a small cluster of blocks:
// block r of C owns the candidates t = r (mod C) with their gains and its
// own part of every list, keeps its own copy of m, and per step exchanges
// one key with the others (st.async into every block's slot, counted on an
// mbarrier there).
#include <string.h>

#include "bf16_dot.cuh"
#include "sgs_gain.cuh"

namespace cp {
namespace {

constexpr int PUSH_CMAX = 16;  // blocks per cluster (16: the non-portable maximum)
constexpr int PUSH_WARPS = 32;
constexpr int PUSH_THREADS = 32 * PUSH_WARPS;

__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint32_t map_rank(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ void hw_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
               : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return done != 0;
}
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
// Chunks load whole, up to 127 entries past a list's end: entries past the
// last list of the buffer.
constexpr size_t LIST_PAD = 128;

// ---------------------------------------------------------------------------
// The first pick of the dense path.  The cost pass's partial sums (g0, one
// per 64-column tile) add the gain's terms in fp32: at most 8 roundings
// inside a tile and one per tile after that, each of relative size 2^-24 of
// non-negative sums, so a total is within 2^-15 (264 x 2^-24 at 256 tiles)
// of the exact sum, which the fixed-point gain differs from by less than
// 2^-23 of it.  Only candidates whose upper bound reaches the largest lower
// bound can be the first pick; their gains are computed exactly.
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
                                                    const float* __restrict__ v_all, int N,
                                                    float m0, int fx,
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
      for (int i0 = lane; i0 < nq; i0 += 8 * 32) {
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

// ---------------------------------------------------------------------------
// The live candidates after the first pick w0, m_j = min(m0, C(w0, j)), and
// every candidate's gain there: one pass over the cost.  A block owns 128
// columns of one owner's rows (t = tl C + rank): tiles of 32 rows x 128
// columns come in by cp.async, four deep; a warp takes 8 of the columns with
// a lane per row (one 16-byte shared load covers four columns), so a
// column's live rows are one ballot, the entries of a list go out
// contiguously and a lane's gain needs no reduction until the tile ends.
// Candidates with nearby indices are near in space, so about half of the
// ballots are empty and skip the arithmetic.  Bound by HBM (the cost read
// once, entries of 8 bytes for the live fifth written).
// List of (j, owner): lists[((bl N + j) C + owner) NC ..], lens alike.
// ---------------------------------------------------------------------------
constexpr int LL_COLS = 128, LL_ROWS = 32, LL_STAGES = 4, LL_WARPS = 16;
constexpr int LL_PITCH = LL_COLS + 4;  // lanes of a 16-byte read (a lane a row) on distinct banks
constexpr int LL_COLS_W = LL_COLS / LL_WARPS;
constexpr size_t LL_SMEM = sizeof(float) * LL_STAGES * LL_ROWS * LL_PITCH;

__global__ void __launch_bounds__(32 * LL_WARPS) k_live_lists(
    const float* __restrict__ cost, int64_t ldc, const float* __restrict__ v_all,
    const gain_t* __restrict__ first, int N, int C, int lgC, int NC, int scene0, float m0, int fx,
    gain_t* __restrict__ gains, Entry* __restrict__ lists, uint32_t* __restrict__ lens) {
  extern __shared__ __align__(16) float s_tile[];  // [LL_STAGES][LL_ROWS][LL_PITCH]
  __shared__ gain_t s_part[2][LL_WARPS][32];
  const int col0 = blockIdx.x * LL_COLS, rank = blockIdx.y, bl = blockIdx.z, b = scene0 + bl;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float* Cb = cost + (size_t)b * N * ldc;
  const float* v = v_all + (size_t)b * N;
  gain_t* G = gains + (size_t)b * N;
  const int nown = N > rank ? (N - rank + C - 1) >> lgC : 0;
  const int ntile = (nown + LL_ROWS - 1) / LL_ROWS;
  const int w0 = key_token(first[b]);
  float m[LL_COLS_W], vj[LL_COLS_W];
  uint32_t cnt[LL_COLS_W];
#pragma unroll
  for (int u = 0; u < LL_COLS_W; ++u) {
    const int j = col0 + LL_COLS_W * w + u;
    m[u] = -INFINITY;  // past the row: nothing is live
    vj[u] = 0.0f;
    cnt[u] = 0u;
    if (j < N) {
      m[u] = fminf(m0, __ldg(Cb + (size_t)w0 * ldc + j));
      vj[u] = __ldg(v + j);
    }
  }
  const size_t lstep = (size_t)C * NC;  // between the lists of adjacent columns
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
            L[u * lstep + cnt[u] + __popc(mask & lt)] =
                make_uint2((uint32_t)tl, __float_as_uint(c[e]));
          }
          cnt[u] += __popc(mask);
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
      if (j < N) lens[((size_t)bl * N + j) * C + rank] = cnt[u];
    }
  }
}

// ---------------------------------------------------------------------------
// The local path's lists: the candidates t with j in M_g(t), by owner block
// (t mod C), and their costs.  One block per scene: counts, an exclusive scan
// and a fill, with counts and cursors in shared memory [N C].  span[(b N + j)
// C + owner] = (offset into the scene's entries, length); the order within a
// list is arbitrary (no result depends on it).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(1024) k_rev_lists(const int32_t* __restrict__ nbr_all,
                                                    const float* __restrict__ slab, int N, int g,
                                                    int kk, int C, int lgC,
                                                    uint2* __restrict__ span_all,
                                                    Entry* __restrict__ ent_all) {
  extern __shared__ int s_c[];  // [N C]
  __shared__ int s_sum[1024];
  const int b = blockIdx.x;
  const int32_t* NB = nbr_all + (size_t)b * N * kk;
  const float* S = slab + (size_t)b * N * g;
  uint2* span = span_all + (size_t)b * N * C;
  Entry* ent = ent_all + (size_t)b * N * g;
  const int64_t ng = (int64_t)N * g;
  const int nc = N * C;
  for (int j = threadIdx.x; j < nc; j += blockDim.x) s_c[j] = 0;
  __syncthreads();
  for (int64_t i = threadIdx.x; i < ng; i += blockDim.x) {
    const int t = (int)(i / g), k = (int)(i % g);
    const int j = k == 0 ? t : NB[(size_t)t * kk + (k - 1)];
    atomicAdd(&s_c[(j << lgC) | (t & (C - 1))], 1);
  }
  __syncthreads();
  // exclusive prefix of the counts: each thread a contiguous chunk, then a
  // scan of the 1024 chunk sums
  const int chunk = (nc + blockDim.x - 1) / blockDim.x;
  const int c0 = min(nc, (int)threadIdx.x * chunk), c1 = min(nc, c0 + chunk);
  int part = 0;
  for (int j = c0; j < c1; ++j) part += s_c[j];
  s_sum[threadIdx.x] = part;
  __syncthreads();
  for (int d = 1; d < (int)blockDim.x; d <<= 1) {
    const int x = threadIdx.x >= (unsigned)d ? s_sum[threadIdx.x - d] : 0;
    __syncthreads();
    s_sum[threadIdx.x] += x;
    __syncthreads();
  }
  int run = s_sum[threadIdx.x] - part;  // the exclusive prefix of this chunk
  for (int j = c0; j < c1; ++j) {
    const int n = s_c[j];
    span[j] = make_uint2((uint32_t)run, (uint32_t)n);
    s_c[j] = run;  // from here on: the next free slot
    run += n;
  }
  __syncthreads();
  for (int64_t i = threadIdx.x; i < ng; i += blockDim.x) {
    const int t = (int)(i / g), k = (int)(i % g);
    const int j = k == 0 ? t : NB[(size_t)t * kk + (k - 1)];
    ent[atomicAdd(&s_c[(j << lgC) | (t & (C - 1))], 1)] =
        make_uint2((uint32_t)(t >> lgC), __float_as_uint(S[i]));
  }
}

// The local path's first gains (m = m0), one warp per candidate.
__global__ void __launch_bounds__(256) k_local_gains(const float* __restrict__ slab,
                                                     const int32_t* __restrict__ nbr,
                                                     const float* __restrict__ v_all, int N, int g,
                                                     int kk, float m0, int fx,
                                                     gain_t* __restrict__ gains) {
  const int t = blockIdx.x * 8 + (threadIdx.x >> 5), b = blockIdx.y, lane = threadIdx.x & 31;
  if (t >= N) return;
  const float* v = v_all + (size_t)b * N;
  const float* srow = slab + ((size_t)b * N + t) * g;
  const int32_t* nb = nbr + ((size_t)b * N + t) * kk;
  gain_t acc = 0ull;
  for (int k = lane; k < g; k += 32) {
    const int j = k == 0 ? t : __ldg(nb + k - 1);
    acc += gain_term(__ldg(v + j), m0, __ldg(srow + k), fx);
  }
  acc = warp_sum_gain(acc);
  if (lane == 0) gains[(size_t)b * N + t] = acc;
}

// ---------------------------------------------------------------------------
// The greedy steps.
// ---------------------------------------------------------------------------
struct PushArgs {
  const float* rows;      // dense: cost [B][N][ldc]; local: slab [B][N][g]
  const int32_t* nbr;     // local: [B][N][kk]
  const float* v;         // [B][N]
  const gain_t* gains0;   // [B][N] gains at the start
  const gain_t* first;    // dense: [B] key of the first pick
  Entry* lists;
  uint32_t* lens;         // dense: [scenes of the wave][N][C]
  uint2* span;            // local: [B][N][C] (offset, length)
  int32_t* order32;       // [B][K]
  float* out_gains;       // [B][K] or null
  double* objective;      // [B] or null
  int* status;
  int64_t ldc;
  uint64_t timeout_ns;
  float m0;
  int fx;
  int N, K, g, kk;
  int C, lgC, NC;         // blocks per cluster (a power of two), its log2, ceil(N / C)
  int lgS;                // log2 of the candidates a warp scans
  int scene0;             // first scene of the wave
  uint32_t off_q, off_lo, off_hi;  // dynamic shared memory offsets
};

// Gains are kept as two 32-bit words (32-bit shared atomics are native); an
// update takes the low word off first and the borrow that its own atomic saw
// with the high word, so the pair is right once every update has run.
template <bool LOCAL>
__global__ void __launch_bounds__(PUSH_THREADS, 1) k_sgs_push(const __grid_constant__ PushArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  float* sm_m = reinterpret_cast<float*>(smem);                     // [ldc or N] coverage cost
  uint32_t* queue = reinterpret_cast<uint32_t*>(smem + a.off_q);    // lowered targets: (k << 16) | j
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
  const int N = a.N, lgC = a.lgC, fx = a.fx;
  const int ncols = LOCAL ? N : (int)a.ldc;
  const int nown = N > rank ? (N - rank + a.C - 1) >> lgC : 0;
  const float* v = a.v + (size_t)b * N;
  const float* R = a.rows + (size_t)b * N * (LOCAL ? (size_t)a.g : (size_t)a.ldc);
  const int32_t* NB = LOCAL ? a.nbr + (size_t)b * N * a.kk : nullptr;
  unsigned long long my_ent = 0ull, my_rows = 0ull;  // list entries (a lane's), rows read

  // state at the start: m, the gains, the first pick (dense)
  int last = -1;  // the last pick, not yet dropped from the candidates
  int start = 0;
  if (!LOCAL) {
    const gain_t f = a.first[b];
    last = key_token(f);
    start = 1;
    if (rank == 0 && threadIdx.x == 0) {
      a.order32[(size_t)b * a.K] = last;
      if (a.out_gains) a.out_gains[(size_t)b * a.K] = key_gain(f);
    }
  }
  for (int j = threadIdx.x; j < ncols; j += PUSH_THREADS) {
    float mj = j < N ? a.m0 : 0.0f;
    if (!LOCAL && j < N) mj = fminf(mj, __ldg(R + (size_t)last * a.ldc + j));
    sm_m[j] = mj;
  }
  for (int tl = threadIdx.x; tl < nown; tl += PUSH_THREADS) {
    const gain_t x = a.gains0[(size_t)b * N + ((tl << lgC) | rank)];
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

  bool ok = true;
  int pref = -1;  // the row last prefetched
  for (int step = start; step < a.K; ++step) {
    const int par = step & 1;
    if (a.C > 1 && threadIdx.x == 0) mbar_expect(&s_bar[par], 8u * (uint32_t)a.C);
    // ---- the warp's best key, when one of its gains changed
    const int ltl = last >> lgC;
    const bool drop = last >= 0 && (last & (a.C - 1)) == rank && ltl >= lo0 && ltl < lo1;
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
      if (lane == 0) s_key[w] = mf ? gain_key(mf - 1u, (mt << lgC) | rank) : 0ull;
    }
    __syncthreads();  // every warp's key is in
    gain_t W = 0ull;
    if (a.C == 1 || w < 2) W = warp_max_key(lane < PUSH_WARPS ? s_key[lane] : 0ull);
    if (a.C > 1) {
      if (w == 0 && lane < a.C)
        st_async_u64(map_rank(smem_addr(&s_res[par][rank]), (uint32_t)lane), W,
                     map_rank(smem_addr(&s_bar[par]), (uint32_t)lane));
      if (!LOCAL && w == 1 && W != 0ull) {  // this block's best row, likely a coming pick's
        const int t = key_token(W);
        if (t != pref && lane == 0) prefetch_l2(R + (size_t)t * a.ldc, (uint32_t)(4 * a.ldc));
        pref = t;
      }
      int good = 1;
      if (lane == 0 && !mbar_test(&s_bar[par], (uint32_t)((step - start) >> 1) & 1u)) {
        const uint64_t t0 = globaltimer_ns();
        uint32_t spins = 0;
        while (!mbar_test(&s_bar[par], (uint32_t)((step - start) >> 1) & 1u)) {
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
    if (pick < 0 || pick >= N) {  // never expected: no candidate left
      if (lane == 0) s_fail = 1;
      if (threadIdx.x == 0 && atomicCAS(a.status, 0, CP_EDEVICE) == 0) {
        a.status[4] = step;
        a.status[5] = b;
        a.status[6] = rank;
        a.status[7] = pick;
      }
    } else {
      if (rank == 0 && threadIdx.x == 0) {
        a.order32[(size_t)b * a.K + step] = pick;
        if (a.out_gains) a.out_gains[(size_t)b * a.K + step] = key_gain(W);
        ++my_rows;
      }
      // ---- S <- S u {t*} (Eq. sgs_update): the targets whose m drops
      if (!LOCAL) {
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
      } else {
        const float* srow = R + (size_t)pick * a.g;
        const int32_t* nb = NB + (size_t)pick * a.kk;
        for (int k = threadIdx.x; k < a.g; k += PUSH_THREADS) {
          const int j = k == 0 ? pick : __ldg(nb + k - 1);
          if (__ldg(srow + k) < sm_m[j])
            queue[atomicAdd(&s_qn, 1)] = ((uint32_t)k << 16) | (uint32_t)j;
        }
      }
    }
    last = pick;
    __syncthreads();  // the lowered targets are listed
    if (s_fail) {     // block-uniform
      ok = false;
      break;
    }
    // ---- two lowered targets a warp at a time: their live candidates lose
    // what the drop took; the entries that stay live are packed to the
    // list's front.  The lists' lengths and first entries load together (an
    // entry past the length is ignored), and four chunks of 32 entries are
    // in flight, their low-word updates issued before any of their results
    // is needed.
    const int qn = s_qn;
    for (int q0 = w; q0 < qn; q0 += 2 * PUSH_WARPS) {
      Entry* L[2];
      uint32_t* len_at[2];
      int j[2], len[2], out[2] = {0, 0};
      float mn[2], vj[2], mo[2];
      Entry x[4];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int qi = q0 + h * PUSH_WARPS;
        const uint32_t e = queue[qi < qn ? qi : q0];
        j[h] = (int)(e & 0xFFFFu);
        const size_t lj = ((size_t)(LOCAL ? b : bl) * N + j[h]) * a.C + rank;
        mn[h] = LOCAL ? __ldg(R + (size_t)pick * a.g + (e >> 16))
                      : __ldg(R + (size_t)pick * a.ldc + j[h]);
        vj[h] = __ldg(v + j[h]);
        mo[h] = sm_m[j[h]];
        if (LOCAL) {
          const uint2 sp = __ldcg(a.span + lj);
          L[h] = a.lists + (size_t)b * N * a.g + sp.x;
          len_at[h] = &a.span[lj].y;
          len[h] = (int)sp.y;
        } else {
          L[h] = a.lists + lj * a.NC;
          len_at[h] = a.lens + lj;
          len[h] = (int)__ldcg(len_at[h]);
        }
        x[2 * h] = __ldcg(L[h] + lane);
        x[2 * h + 1] = __ldcg(L[h] + 32 + lane);
        if (qi >= qn) len[h] = 0;
      }
      // chunks x[0..3]: entry i[u] + lane of list h[u]
      auto apply = [&](const int (&hh)[4], const int (&i0)[4]) {
        gain_t d[4];
        uint32_t old[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int h = hh[u];
          const float c = __uint_as_float(x[u].y);
          d[u] = i0[u] + lane < len[h] ? gain_term(vj[h], mo[h], c, fx) - gain_term(vj[h], mn[h], c, fx)
                                       : 0ull;
          old[u] = 0u;
          if (d[u] != 0ull) old[u] = atomicAdd(g_lo + x[u].x, 0u - (uint32_t)d[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int h = hh[u];
          if (d[u] != 0ull) {
            const uint32_t dh = (uint32_t)(d[u] >> 32) + (old[u] < (uint32_t)d[u] ? 1u : 0u);
            if (dh) atomicAdd(g_hi + x[u].x, 0u - dh);
            s_dirty[x[u].x >> a.lgS] = 1u;
          }
          if (i0[u] < len[h]) {  // warp-uniform
            const int i = i0[u] + lane;
            const bool stay = i < len[h] && __uint_as_float(x[u].y) < mn[h];
            const uint32_t mask = __ballot_sync(0xFFFFFFFFu, stay);
            const int p = out[h] + __popc(mask & ((1u << lane) - 1u));
            if (stay && p != i) __stcg(L[h] + p, x[u]);
            out[h] += __popc(mask);
          }
        }
      };
      apply({0, 0, 1, 1}, {0, 32, 0, 32});
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        for (int i0 = 64; i0 < len[h]; i0 += 128) {
#pragma unroll
          for (int u = 0; u < 4; ++u) x[u] = __ldcg(L[h] + i0 + 32 * u + lane);
          if (h == 0)
            apply({0, 0, 0, 0}, {i0, i0 + 32, i0 + 64, i0 + 96});
          else
            apply({1, 1, 1, 1}, {i0, i0 + 32, i0 + 64, i0 + 96});
        }
        if (lane == 0 && len[h]) {
          my_ent += (unsigned long long)len[h];
          if (out[h] != len[h]) __stcg(len_at[h], (uint32_t)out[h]);
        }
        if (lane == 0) sm_m[j[h]] = mn[h];
      }
    }
    __syncthreads();  // gains and m are settled
    if (threadIdx.x == 0) s_qn = 0;
  }

  unsigned long long* cstats = reinterpret_cast<unsigned long long*>(
      reinterpret_cast<unsigned char*>(a.status) + kCallStatsOffset);
  if (lane == 0 && my_ent) {
    atomicAdd(&cstats[0], my_ent);
    atomicAdd(&cstats[2], 8ull * my_ent);
  }
  if (rank == 0 && threadIdx.x == 0) {
    atomicAdd(&cstats[1], (unsigned long long)a.K);
    atomicAdd(&cstats[2], my_rows * (LOCAL ? 8ull * (unsigned long long)a.g
                                           : 4ull * (unsigned long long)ncols));
  }
  __syncthreads();
  if (ok && rank == 0 && a.objective) {
    const double F = objective_sum(sm_m, v, N);
    if (threadIdx.x == 0) a.objective[b] = F;
  }
  if (!ok) {  // a peer's last key may still be on its way here: let it land
    const uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 500000ull) {
    }
  }
  hw_cluster_sync();  // nobody leaves while a peer may still write to its shared memory
}

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

// Scenes whose lists are held at once.  A dense scene's lists take 8 N^2
// bytes at their largest (twice its cost), so a large batch runs in waves:
// as many scenes as fit 24 GB less a twelfth of the whole cost, at least one.
int64_t push_wave(int64_t B, int64_t N, int64_t ldc) {
  const double per = 8.0 * (double)N * (double)(N + PUSH_CMAX);
  const double room = 24.0e9 - 4.0 * (double)B * (double)N * (double)ldc / 12.0;
  const int64_t w = room > per ? (int64_t)(room / per) : 1;
  return w < B ? w : B;
}

struct PushPlan {
  size_t gains, first, max_bits, zero_bytes, sums, lens, lists, total;
  int64_t wave;
};
PushPlan push_plan(int64_t B, int64_t N, int64_t g, int64_t ldc) {
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
    p.lens = take(sizeof(uint2) * BN * PUSH_CMAX);
    p.lists = take(sizeof(Entry) * (BN * (size_t)g + LIST_PAD));
  } else {
    p.first = take(sizeof(gain_t) * (size_t)B);
    p.max_bits = take(sizeof(uint32_t) * (size_t)B);
    p.zero_bytes = off;
    p.sums = take(sizeof(float) * BN);
    p.wave = push_wave(B, N, ldc);
    p.lens = take(sizeof(uint32_t) * (size_t)p.wave * (size_t)N * PUSH_CMAX);
    p.lists =
        take(sizeof(Entry) * ((size_t)p.wave * (size_t)N * (size_t)(N + PUSH_CMAX) + LIST_PAD));
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
  a.off_lo = a.off_q + (uint32_t)(sizeof(uint32_t) * (size_t)(a.g < a.N ? a.g : a.N));
  a.off_lo = (a.off_lo + 15u) & ~15u;
  a.off_hi = a.off_lo + (uint32_t)(sizeof(uint32_t) * (size_t)a.NC);
  return a.off_hi + sizeof(uint32_t) * (size_t)a.NC;
}

// The largest cluster, C0 halved as often as needed, that the device can
// hold; its launch configuration in cfg (attr must outlive it).
template <bool LOCAL>
int push_config(PushArgs& a, int C0, int64_t scenes, int64_t ncols, const DeviceInfo& di,
                cudaStream_t s, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr) {
  auto fn = k_sgs_push<LOCAL>;
  for (int C = C0; C >= 1; C >>= 1) {
    const size_t smem = push_shape(a, C, ncols);
    if (smem + 2048 > (size_t)di.max_smem_optin) continue;
    if (cuda_status(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem),
                    "launch_sgs_push: smem attribute") != CP_OK)
      return CP_ECUDA;
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

}  // namespace

// One size for every neighbourhood: a workspace of these sizes serves the
// dense path and each local one.
size_t sgs_push_ws_bytes(int64_t B, int64_t N, int64_t g, int64_t ldc) {
  const size_t dense = push_plan(B, N, N, ldc).total;
  const size_t local = g < N ? push_plan(B, N, g, ldc).total : 0;
  return local > dense ? local : dense;
}

int launch_sgs_push(const float* cost, int64_t ldc, const float* slab, const int32_t* nbr,
                    const float* v, const DevParams& P, int64_t B, int64_t N, int64_t K,
                    int32_t* order32, float* gains, double* objective, int* status,
                    cudaStream_t s, const float* g0, void* ws) {
  DeviceInfo di;
  if (device_info(&di) != CP_OK) return CP_ECUDA;
  const bool local = P.g < N;
  const PushPlan pl = push_plan(B, N, P.g, ldc);
  unsigned char* base = static_cast<unsigned char*>(ws);
  gain_t* gains64 = reinterpret_cast<gain_t*>(base + pl.gains);
  const int fx = gain_fx(P.m0);
  PushArgs a{};
  a.rows = local ? slab : cost;
  a.nbr = nbr;
  a.v = v;
  a.gains0 = gains64;
  a.order32 = order32;
  a.out_gains = gains;
  a.objective = objective;
  a.status = status;
  a.ldc = ldc;
  a.timeout_ns = P.timeout_ns;
  a.m0 = P.m0;
  a.fx = fx;
  a.N = (int)N;
  a.K = (int)K;
  a.g = P.g;
  a.kk = P.kk;
  a.lists = reinterpret_cast<Entry*>(base + pl.lists);
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  if (local) {
    const int C0 = N > 12288 ? 2 : 1;
    CP_TRY_STATUS(push_config<true>(a, C0, B, N, di, s, &cfg, attr));
    a.span = reinterpret_cast<uint2*>(base + pl.lens);
    const size_t rsmem = sizeof(int) * (size_t)N * (size_t)a.C;
    if (rsmem > 40 * 1024 &&
        cuda_status(cudaFuncSetAttribute(k_rev_lists, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)rsmem),
                    "launch_sgs_push: reverse-list smem attribute") != CP_OK)
      return CP_ECUDA;
    k_rev_lists<<<(unsigned)B, 1024, rsmem, s>>>(nbr, slab, (int)N, P.g, P.kk, a.C, a.lgC, a.span,
                                                 a.lists);
    CP_TRY_STATUS(last_launch_status());
    k_local_gains<<<dim3((unsigned)((N + 7) / 8), (unsigned)B), 256, 0, s>>>(
        slab, nbr, v, (int)N, P.g, P.kk, P.m0, fx, gains64);
    CP_TRY_STATUS(last_launch_status());
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_sgs_push<true>, a);
    note_launch();
    return cuda_status(e, "launch_sgs_push: local");
  }
  gain_t* first = reinterpret_cast<gain_t*>(base + pl.first);
  uint32_t* max_bits = reinterpret_cast<uint32_t*>(base + pl.max_bits);
  float* sums = g0 ? reinterpret_cast<float*>(base + pl.sums) : nullptr;
  a.first = first;
  a.lens = reinterpret_cast<uint32_t*>(base + pl.lens);
  CP_TRY_STATUS(cuda_status(cudaMemsetAsync(base + pl.gains, 0, pl.zero_bytes, s),
                            "launch_sgs_push: gains"));
  if (g0) {
    k_first_bounds<<<dim3((unsigned)((N + 255) / 256), (unsigned)B), 256, 0, s>>>(
        g0, fst_apply_slots(ldc), (int)N, sums, max_bits);
    CP_TRY_STATUS(last_launch_status());
  }
  const int64_t groups = g0 ? (N + 255) / 256 : (N + 7) / 8;
  k_first_pick<<<dim3((unsigned)(groups < 512 ? groups : 512), (unsigned)B), 256, 0, s>>>(
      cost, ldc, v, (int)N, P.m0, fx, sums, max_bits, first);
  CP_TRY_STATUS(last_launch_status());
  if (cuda_status(cudaFuncSetAttribute(k_live_lists, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)LL_SMEM),
                  "launch_sgs_push: lists smem attribute") != CP_OK)
    return CP_ECUDA;
  for (int64_t b0 = 0; b0 < B; b0 += pl.wave) {
    const int64_t nb = B - b0 < pl.wave ? B - b0 : pl.wave;
    int C0 = PUSH_CMAX;
    while (C0 > 1 && ((int64_t)C0 * nb > di.sm_count || N / C0 < 256)) C0 >>= 1;
    if (C0 < 2 && N > 12288) C0 = 2;
    CP_TRY_STATUS(push_config<false>(a, C0, nb, ldc, di, s, &cfg, attr));
    a.scene0 = (int)b0;
    if (K > 1) {
      k_live_lists<<<dim3((unsigned)((N + LL_COLS - 1) / LL_COLS), (unsigned)a.C, (unsigned)nb),
                     32 * LL_WARPS, LL_SMEM, s>>>(cost, ldc, v, first, (int)N, a.C, a.lgC, a.NC,
                                                  (int)b0, P.m0, fx, gains64, a.lists, a.lens);
      CP_TRY_STATUS(last_launch_status());
    }
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_sgs_push<false>, a);
    note_launch();
    CP_TRY_STATUS(cuda_status(e, "launch_sgs_push: dense"));
  }
  return CP_OK;
}

}  // namespace cp
