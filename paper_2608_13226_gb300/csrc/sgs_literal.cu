// K5 as Sec. 3.5 prints it (sgs_mode 2): Eqs. srpot_sinkhorn, greedy_flow,
// sgs_select and sgs_update read word for word.
//
// At greedy step l the selected tokens s_0 .. s_{l-1} are the sources of an
// entropic semi-relaxed OT (Eq. srpot_sinkhorn), each with mass 1/K, and
// every token is a target with capacity v_j.  Its plan has the Gibbs form
// P_ij = exp((f_i + g_j - C(s_i, j)) / eps) with g <= 0, and block
// coordinate ascent on the dual alternates
//   rows:    f_i = eps log(1/K) - eps LSE_j((g_j - C(s_i, j)) / eps)   (P 1 = u)
//   columns: g_j = min(0, eps log v_j - eps LSE_i((f_i - C(s_i, j)) / eps))
//            (the capacity cap P^T 1 <= v; a column below it keeps g_j = 0)
// for sot_iters iterations, the column potentials carried over from step
// l-1 (zeros at l = 1).  The residual capacity (Eq. greedy_flow) is
//   r_j = max(v_j - sum_i P_ij, 0)     (r = v at l = 0),
// and the next token minimises the residual-weighted local cost (Eq.
// sgs_select)  score(t) = sum_{j in M_g(t)} r_j C(t, j)  over the
// unselected tokens, lowest index on equal scores.
//
// While the l selected rows fit the shared memory of a cluster of blocks, a
// step is two launches: its iterations (k_lit_sinkhorn) and the scores.  One
// scene of 1024 tokens, 102 picks, 20 iterations a step: 4.6 ms, of which the
// iterations take ~1.6 us each, bound by their chain of latencies; one launch
// a phase and iteration, the form before, took 21.7.  Beyond that the path is
// bound by L2 and HBM: each iteration reads the l selected rows of the
// dense cost twice (rows, then columns), the score reads every candidate's
// row once.  One launch per phase covers all B scenes: columns a thread per
// target column (the l source indices and potentials staged in shared
// memory, the cost read coalesced along the row; a block spreads 32 columns
// over 16 groups of source rows), rows a block per source row, scores a warp
// per candidate; every thread keeps eight loads in flight.  Each step's winner is the smallest
// (score bits, index) key, reduced with one 64-bit atomicMin per block into
// that step's slot (initialised to all ones), so no separate argmin pass
// runs; non-negative floats order like their bit patterns, and every score
// is a sum of products of non-negative numbers.  Log-sum-exp is accumulated
// online (the running maximum rescales the running sum only when it grows).
#include "common.cuh"

namespace cp {
namespace {

constexpr int LIT_THREADS = 256;

struct Lse {
  float m, s;  // running maximum and sum of exp(x - m)
};
__device__ __forceinline__ void lse_add(Lse& a, float x) {
  if (x > a.m) {
    a.s = a.s * expf(a.m - x) + 1.0f;  // expf(-inf) = 0 on the first finite term
    a.m = x;
  } else if (x > -INFINITY) {
    a.s += expf(x - a.m);
  }
}
__device__ __forceinline__ Lse lse_merge(Lse a, Lse b) {
  if (a.m < b.m) {
    const Lse t = a;
    a = b;
    b = t;
  }
  if (b.m > -INFINITY) a.s += b.s * expf(b.m - a.m);
  return a;
}
__device__ __forceinline__ float lse_value(const Lse& a) {
  return a.m > -INFINITY ? a.m + logf(a.s) : -INFINITY;
}
__device__ __forceinline__ Lse warp_lse(Lse a) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    Lse b;
    b.m = __shfl_xor_sync(0xFFFFFFFFu, a.m, o);
    b.s = __shfl_xor_sync(0xFFFFFFFFu, a.s, o);
    a = lse_merge(a, b);
  }
  return a;
}
__device__ __forceinline__ int key_index(unsigned long long k) {
  return (int)(uint32_t)(k & 0xFFFFFFFFull);
}

// Row potentials of the l sources: f_i = eps log u - eps LSE_j((g_j - C_ij) / eps).
// One block per source row: thread x takes the columns x, x + 256, ...,
// eight loads in flight before their terms are added in column order; the
// threads' partial log-sum-exps merge in a fixed order (warps by butterfly,
// then the 8 warps in order).
__global__ void __launch_bounds__(LIT_THREADS) k_lit_rows(
    const float* __restrict__ C, int64_t ldc, int N, int K, int l,
    const unsigned long long* __restrict__ keys, const float* __restrict__ gpot, float eps,
    float inv_eps, float log_u, float* __restrict__ fpot) {
  __shared__ float s_m[LIT_THREADS / 32], s_s[LIT_THREADS / 32];
  const int b = blockIdx.y, i = blockIdx.x;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int s = key_index(keys[(size_t)b * K + i]);
  const float* row = C + ((size_t)b * N + s) * ldc;
  const float* g = gpot + (size_t)b * N;
  Lse a{-INFINITY, 0.0f};
  for (int j0 = threadIdx.x; j0 < N; j0 += 8 * LIT_THREADS) {
    float x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int j = j0 + u * LIT_THREADS;
      x[u] = j < N ? (__ldg(g + j) - __ldg(row + j)) * inv_eps : -INFINITY;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) lse_add(a, x[u]);
  }
  a = warp_lse(a);
  if (lane == 0) {
    s_m[w] = a.m;
    s_s[w] = a.s;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    Lse t{s_m[0], s_s[0]};
    for (int q = 1; q < LIT_THREADS / 32; ++q) t = lse_merge(t, Lse{s_m[q], s_s[q]});
    fpot[(size_t)b * K + i] = eps * (log_u - lse_value(t));
  }
}

// Per target column j, LSE_i((f_i - C(s_i, j)) / eps) over the l sources.
// A block takes 32 columns (threadIdx.x) and splits the sources over 16 row
// groups (threadIdx.y: i = y, y + 16, ...), each warp reading 128
// contiguous bytes of a source row; the 16 partial log-sum-exps of a column
// merge in a fixed order.  RESID = false: the column potential g_j (the
// capacity cap).  RESID = true: the residual r_j = max(v_j - exp(g_j / eps +
// LSE), 0), and block 0 marks the previous step's pick as selected.
constexpr int LC_COLS = 32, LC_GROUPS = 16, LC_CHUNK = 256;
template <bool RESID>
__global__ void __launch_bounds__(LC_COLS * LC_GROUPS) k_lit_cols(
    const float* __restrict__ C, int64_t ldc, int N, int K, int l,
    const unsigned long long* __restrict__ keys, const float* __restrict__ fpot,
    const float* __restrict__ v, float eps, float inv_eps, float* __restrict__ gpot,
    float* __restrict__ resid, uint8_t* __restrict__ chosen) {
  __shared__ int s_idx[LC_CHUNK];
  __shared__ float s_f[LC_CHUNK];
  __shared__ float s_m[LC_GROUPS][LC_COLS], s_s[LC_GROUPS][LC_COLS];
  const int b = blockIdx.y;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int tid = ty * LC_COLS + tx;
  const int j = blockIdx.x * LC_COLS + tx;
  if (RESID && l > 0 && blockIdx.x == 0 && tid == 0)
    chosen[(size_t)b * N + key_index(keys[(size_t)b * K + l - 1])] = 1;
  const float* Cb = C + (size_t)b * N * ldc;
  Lse a{-INFINITY, 0.0f};
  for (int i0 = 0; i0 < l; i0 += LC_CHUNK) {
    const int n = min(LC_CHUNK, l - i0);
    __syncthreads();  // the previous chunk is consumed
    if (tid < n) {
      s_idx[tid] = key_index(keys[(size_t)b * K + i0 + tid]);
      s_f[tid] = fpot[(size_t)b * K + i0 + tid];
    }
    __syncthreads();
    if (j < N)
      for (int i1 = ty; i1 < n; i1 += 8 * LC_GROUPS) {  // eight loads in flight
        float x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int ii = i1 + u * LC_GROUPS;
          x[u] = ii < n ? (s_f[ii] - __ldg(Cb + (size_t)s_idx[ii] * ldc + j)) * inv_eps
                        : -INFINITY;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) lse_add(a, x[u]);
      }
  }
  s_m[ty][tx] = a.m;
  s_s[ty][tx] = a.s;
  __syncthreads();
  if (ty != 0 || j >= N) return;
  for (int q = 1; q < LC_GROUPS; ++q) a = lse_merge(a, Lse{s_m[q][tx], s_s[q][tx]});
  const float vj = v[(size_t)b * N + j];
  if (!RESID) {
    gpot[(size_t)b * N + j] = vj > 0.0f ? fminf(0.0f, eps * (logf(vj) - lse_value(a))) : -INFINITY;
  } else {
    const float gj = l > 0 ? gpot[(size_t)b * N + j] : 0.0f;
    const float lv = lse_value(a);
    const float col = (lv > -INFINITY && gj > -INFINITY) ? expf(gj * inv_eps + lv) : 0.0f;
    resid[(size_t)b * N + j] = fmaxf(vj - col, 0.0f);
  }
}

// All Sinkhorn iterations of a step and its residual in one launch, while the
// l selected rows fit the shared memory of a cluster: block r of the cluster
// holds columns [r W, (r + 1) W) of every selected row, their potentials and
// capacities.  A row's sum over all columns is the blocks' partial ones,
// which every block copies into every block (one bulk copy each, counted on
// an mbarrier there; two buffers in turn: a block that sends into one again
// has seen the answer to the other, so everybody is done with it); the
// columns are the block's own.
//
// The iterations run on the factors of the plan, P_ij = F_i E_ij G_j with
// E = exp(-C / eps) formed once (to a few ulp: the argument in two parts), F = exp(f / eps) = (1 / K) / sum_j E_ij G_j and G = exp(g /
// eps) = min(1, v_j / sum_i F_i E_ij): a multiply-add a term, no exponential
// and no logarithm.  Nothing over- or underflows while C <= 80 eps and a row's
// sum is at least 2^-80 (F <= 2^80; a flushed product is below 2^-126, 2^-46
// of the sum); a column's sum may be smaller where v_j is not, G_j being 1
// then.  A step that leaves this range (E's argument, a row's sum, a column's
// or a G below 2^-110) runs again on the potentials themselves, with
// log-sum-exps of (g - C) and (f - C); a pair (maximum, sum) a row and block
// is then exchanged instead of a sum.
//
// What bounds an iteration is its chain: row terms, exchange, column terms.
// 8 or 16 lanes take a row (16-byte shared loads), 8 a column; the row pitch
// is 4 mod 32, so that the column reads (8 rows x 4 columns a warp) fall into
// distinct banks too.
constexpr int LS_THREADS = 512;
struct SinkArgs {
  const float* C;
  const unsigned long long* keys;
  const float* v;
  float* gpot;
  float* resid;
  uint8_t* chosen;
  int64_t ldc;
  int N, K, l, iters;
  int CB, W, pitch;   // blocks a cluster, columns a block, row pitch
  int lp;             // pitch of a block's pairs, at least l
  float eps, inv_eps, inv_eps_lo, k, eps_log_u, u;
  int* status;
  uint64_t timeout_ns;
};

// A log-sum-exp of x / eps here: m the largest x (a cost), s the sum of
// exp((x - m) / eps); k = log2(e) / eps.  x - m of the terms that matter is
// small, so 2^((x - m) k) loses less than exp(x / eps - m / eps) does.
__device__ __forceinline__ float sink_exp(float x, float m, float k) {
  float r;  // m is finite, x may be -inf
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"((x - m) * k));
  return x > -INFINITY ? r : 0.0f;
}
__device__ __forceinline__ float finite_or_0(float m) { return m > -INFINITY ? m : 0.0f; }
// Over the lanes that differ in the bits FIRST .. LAST / 2.
template <int FIRST, int LAST>
__device__ __forceinline__ Lse lanes_lse(Lse a, float k) {
  float m = a.m;
#pragma unroll
  for (int o = FIRST; o < LAST; o <<= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
  float s = a.s * sink_exp(a.m, finite_or_0(m), k);
#pragma unroll
  for (int o = FIRST; o < LAST; o <<= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
  return Lse{m, s};
}
// Adds four terms.
__device__ __forceinline__ void lse_add4(Lse& a, float x0, float x1, float x2, float x3, float k) {
  const float m = fmaxf(fmaxf(fmaxf(x0, x1), fmaxf(x2, x3)), a.m), base = finite_or_0(m);
  a.s = a.s * sink_exp(a.m, base, k) + ((sink_exp(x0, base, k) + sink_exp(x1, base, k)) +
                                        (sink_exp(x2, base, k) + sink_exp(x3, base, k)));
  a.m = m;
}

// A block's partial log-sum-exps of the rows staged in S, LPR lanes a row.
template <int LPR>
__device__ __forceinline__ void sink_rows(const SinkArgs& a, const float* S, const float* g,
                                          float2* mine) {
  constexpr int ROWS = LS_THREADS / LPR;  // a turn of the block
  const int sub = threadIdx.x & (LPR - 1), first = threadIdx.x / LPR;
  for (int i0 = 0; i0 < a.l; i0 += ROWS) {
    if (i0 + first - (int)(threadIdx.x & 31) / LPR >= a.l) break;  // warp-uniform
    const int i = i0 + first;
    const float* row = S + (size_t)min(i, a.l - 1) * a.pitch;
    Lse x{-INFINITY, 0.0f};
#pragma unroll 2
    for (int j0 = 0; j0 < a.W; j0 += 4 * LPR) {
      const int j = j0 + 4 * sub;
      const bool in = j < a.W;
      const float4 c = in ? *reinterpret_cast<const float4*>(row + j) : make_float4(0, 0, 0, 0);
      const float4 p = in ? *reinterpret_cast<const float4*>(g + j)
                          : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
      lse_add4(x, p.x - c.x, p.y - c.y, p.z - c.z, p.w - c.w, a.k);
    }
    x = lanes_lse<1, LPR>(x, a.k);
    if (sub == 0 && i < a.l) mine[i] = make_float2(x.m, x.s);
  }
}
// Row potentials from every block's pairs.
template <int LPR>
__device__ __forceinline__ void sink_join(const SinkArgs& a, const float2* all, float* f) {
  constexpr int ROWS = LS_THREADS / LPR;
  const int sub = threadIdx.x & (LPR - 1), first = threadIdx.x / LPR;
  for (int i0 = 0; i0 < a.l; i0 += ROWS) {
    if (i0 + first - (int)(threadIdx.x & 31) / LPR >= a.l) break;  // warp-uniform
    const int i = i0 + first;
    float2 y[16 / LPR];
    float m = -INFINITY;
#pragma unroll
    for (int u = 0; u < 16 / LPR; ++u) {
      const int r = sub + LPR * u;
      y[u] = r < a.CB && i < a.l ? all[(size_t)r * a.lp + i] : make_float2(-INFINITY, 0.0f);
      m = fmaxf(m, y[u].x);
    }
    Lse x{m, 0.0f};
#pragma unroll
    for (int u = 0; u < 16 / LPR; ++u) x.s += y[u].y * sink_exp(y[u].x, finite_or_0(m), a.k);
    x = lanes_lse<1, LPR>(x, a.k);
    if (sub == 0 && i < a.l) f[i] = a.eps_log_u - (x.m + a.eps * logf(x.s));
  }
}

// The same on the factors: sums of E_ij G_j.
template <int LPR>
__device__ __forceinline__ void factor_rows(const SinkArgs& a, const float* E, const float* G,
                                            float* mine) {
  constexpr int ROWS = LS_THREADS / LPR;
  const int sub = threadIdx.x & (LPR - 1), first = threadIdx.x / LPR;
  for (int i0 = 0; i0 < a.l; i0 += ROWS) {
    if (i0 + first - (int)(threadIdx.x & 31) / LPR >= a.l) break;  // warp-uniform
    const int i = i0 + first;
    const float* row = E + (size_t)min(i, a.l - 1) * a.pitch;
    float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f, s3 = 0.0f;
#pragma unroll 2
    for (int j = 4 * sub; j < a.W; j += 4 * LPR) {
      const float4 e = *reinterpret_cast<const float4*>(row + j);
      const float4 p = *reinterpret_cast<const float4*>(G + j);
      s0 = fmaf(e.x, p.x, s0);
      s1 = fmaf(e.y, p.y, s1);
      s2 = fmaf(e.z, p.z, s2);
      s3 = fmaf(e.w, p.w, s3);
    }
    float s = (s0 + s1) + (s2 + s3);
#pragma unroll
    for (int o = 1; o < LPR; o <<= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    if (sub == 0 && i < a.l) mine[i] = s;
  }
}

__global__ void __launch_bounds__(LS_THREADS, 1) k_lit_sinkhorn(const __grid_constant__ SinkArgs a) {
  extern __shared__ __align__(16) float sm[];
  const int l = a.l, W = a.W, pitch = a.pitch, lp = a.lp;
  float* S = sm;                                        // [l][pitch] E, or C
  float* g = S + (size_t)l * pitch;                     // [W] G, or g
  float2* mine = reinterpret_cast<float2*>(g + W);      // [2][lp] this block's sums, or pairs
  float2* all = mine + 2 * lp;                          // [2][CB][lp] every block's
  float* cap = reinterpret_cast<float*>(all + (size_t)2 * a.CB * lp);  // [W] v, or eps log v
  float* f = cap + W;                                                // [l] F, or f
  __shared__ __align__(8) uint64_t s_bar[2];
  __shared__ int s_fail, s_bad, s_again, s_abort;
  const int rank = (int)cluster_ctarank(), b = blockIdx.x / a.CB;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c0 = rank * W, nc = max(0, min(W, a.N - c0));
  const unsigned long long* keys = a.keys + (size_t)b * a.K;
  if (threadIdx.x == 0) {
    if (rank == 0) a.chosen[(size_t)b * a.N + key_index(keys[l - 1])] = 1;
    s_fail = s_bad = s_again = s_abort = 0;
    mbar_init(&s_bar[0], 1);
    mbar_init(&s_bar[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  bool ok = true;
  int turn = 0;
  for (int form = 0; form < 2 && ok; ++form) {
    const bool factors = form == 0;
    bool bad = false;  // out of the factors' range
    for (int j = threadIdx.x; j < W; j += LS_THREADS) {
      const size_t gj = (size_t)b * a.N + c0 + j;
      const float vj = j < nc ? __ldg(a.v + gj) : 0.0f, pj = j < nc ? a.gpot[gj] : -INFINITY;
      if (factors) {
        const float x = pj * a.inv_eps;
        bad |= x < -76.0f && pj > -INFINITY;
        g[j] = expf(x);
        cap[j] = vj;
      } else {
        g[j] = pj;
        cap[j] = vj > 0.0f ? a.eps * logf(vj) : -INFINITY;
      }
    }
    // the rows, 16 bytes a thread and turn; four turns' loads in flight
    const int tpr = W >> 2, nq = l * tpr;
    for (int q0 = threadIdx.x; q0 < nq; q0 += 4 * LS_THREADS) {
      float4 c[4];
      int at[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int q = min(q0 + u * LS_THREADS, nq - 1), i = q / tpr, j = 4 * (q - i * tpr);
        at[u] = i * pitch + j;
        // rows are padded to a multiple of four
        c[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (j < nc)
          c[u] = __ldg(reinterpret_cast<const float4*>(
              a.C + ((size_t)b * a.N + key_index(__ldg(keys + i))) * a.ldc + c0 + j));
        if (j + 1 >= nc) c[u].y = 0.0f;
        if (j + 2 >= nc) c[u].z = 0.0f;
        if (j + 3 >= nc) c[u].w = 0.0f;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (factors) {
          float* e = &c[u].x;
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            const float x = e[h] * a.inv_eps;
            const float lo = fmaf(e[h], a.inv_eps, -x) + e[h] * a.inv_eps_lo;
            bad |= !(x <= 80.0f);
            e[h] = expf(-x) * (1.0f - lo);
          }
        }
        if (q0 + u * LS_THREADS < nq) *reinterpret_cast<float4*>(S + at[u]) = c[u];
      }
    }
    hw_cluster_sync();  // every block's barriers are set up, and its columns are staged
    const uint32_t bytes = factors ? 4u * (uint32_t)((l + 3) & ~3) : 8u * (uint32_t)((l + 1) & ~1);
    for (int it = 0; it < a.iters; ++it, ++turn) {
      const int buf = turn & 1;
      const uint32_t parity = (uint32_t)(turn >> 1) & 1u;
      if (factors) {
        if (l > LS_THREADS / 16)
          factor_rows<8>(a, S, g, reinterpret_cast<float*>(mine + buf * lp));
        else
          factor_rows<16>(a, S, g, reinterpret_cast<float*>(mine + buf * lp));
      } else {
        if (l > LS_THREADS / 16)
          sink_rows<8>(a, S, g, mine + buf * lp);
        else
          sink_rows<16>(a, S, g, mine + buf * lp);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncthreads();  // the block's sums are complete
      float2* got = all + (size_t)buf * a.CB * lp;
      if (w < a.CB && lane == 0) {  // one copy a warp: a warp issues its lanes' one after the other
        if (w == 0) mbar_expect(&s_bar[buf], bytes * (uint32_t)a.CB);
        asm volatile(
            "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], "
            "%2, [%3];" ::"r"(map_rank(smem_addr(got + (size_t)rank * lp), (uint32_t)w)),
            "r"(smem_addr(mine + buf * lp)), "r"(bytes),
            "r"(map_rank(smem_addr(&s_bar[buf]), (uint32_t)w))
            : "memory");
      }
      int good = 1;
      if (lane == 0 && !mbar_test(&s_bar[buf], parity)) {
        const uint64_t t0 = globaltimer_ns();
        uint32_t spins = 0;
        while (!mbar_test(&s_bar[buf], parity)) {
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
      if (good) {
        if (factors) {
          for (int i = threadIdx.x; i < l; i += LS_THREADS) {
            float y[16];
#pragma unroll
            for (int r = 0; r < 16; ++r)
              y[r] = r < a.CB ? reinterpret_cast<const float*>(got + (size_t)r * lp)[i] : 0.0f;
            float s = 0.0f;
#pragma unroll
            for (int r = 0; r < 16; ++r) s += y[r];
            bad |= !(s >= 8.2718061e-25f && s <= 3.0e38f);  // 2^-80
            f[i] = a.u / s;
          }
        } else if (l > LS_THREADS / 16) {
          sink_join<8>(a, got, f);
        } else {
          sink_join<16>(a, got, f);
        }
      }
      __syncthreads();
      if (s_fail) {  // block-uniform
        ok = false;
        break;
      }
      // columns: 4 a warp, 8 lanes each
      const int sub = lane >> 2;
      for (int j0 = 4 * w; j0 < nc; j0 += LS_THREADS / 8) {
        const int j = j0 + (lane & 3);
        const float* col = S + min(j, nc - 1);
        const size_t gj = (size_t)b * a.N + c0 + j;
        if (factors) {
          float s0 = 0.0f, s1 = 0.0f;
          int i = sub;
#pragma unroll 4
          for (; i + 8 < l; i += 16) {
            s0 = fmaf(f[i], col[i * pitch], s0);
            s1 = fmaf(f[i + 8], col[(i + 8) * pitch], s1);
          }
          if (i < l) s0 = fmaf(f[i], col[i * pitch], s0);
          float s = s0 + s1;
          s += __shfl_xor_sync(0xFFFFFFFFu, s, 4);
          s += __shfl_xor_sync(0xFFFFFFFFu, s, 8);
          s += __shfl_xor_sync(0xFFFFFFFFu, s, 16);
          if (sub == 0 && j < nc) {
            const float vj = cap[j], p = vj > 0.0f ? fminf(1.0f, vj / s) : 0.0f;
            // (2^-80, 2^-60, 2^-110)
            bad |= !(s >= 8.2718061e-25f || vj >= 8.6736174e-19f || vj == 0.0f) ||
                   !(p >= 7.7037198e-34f || vj == 0.0f);
            g[j] = p;
            if (it == a.iters - 1) {
              // a column at its capacity leaves nothing (v - (v / s) s would
              // leave its rounding)
              a.resid[gj] = p < 1.0f ? 0.0f : fmaxf(vj - s, 0.0f);
              cap[j] = p > 0.0f ? a.eps * logf(p) : -INFINITY;  // the potential to carry on
            }
          }
        } else {
          Lse x{-INFINITY, 0.0f};
#pragma unroll 2
          for (int i0 = 0; i0 < l; i0 += 32) {
            float t[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int i = i0 + sub + 8 * u;
              t[u] = i < l ? f[i] - col[i * pitch] : -INFINITY;
            }
            lse_add4(x, t[0], t[1], t[2], t[3], a.k);
          }
          x = lanes_lse<4, 32>(x, a.k);
          if (sub == 0 && j < nc) {
            const float lv = x.m + a.eps * logf(x.s), ev = cap[j];
            const float p = ev > -INFINITY ? fminf(0.0f, ev - lv) : -INFINITY;
            g[j] = p;
            if (it == a.iters - 1) {
              const float sum = lv > -INFINITY ? expf(lv * a.inv_eps) : 0.0f;
              a.resid[gj] = p < 0.0f ? 0.0f : fmaxf(__ldg(a.v + gj) - sum, 0.0f);
            }
          }
        }
      }
      __syncthreads();
    }
    if (bad) s_bad = 1;
    if (!ok) {  // a peer's copy may still be on its way here, or one of ours read: let them land
      const uint64_t t0 = globaltimer_ns();
      while (globaltimer_ns() - t0 < 500000ull) {
      }
    }
    __syncthreads();
    // one block's step again is everybody's, and so is its giving up: a block
    // may have passed the wait that another one gave up in
    if ((!ok || (factors && s_bad)) && threadIdx.x < a.CB)
      asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(
                       map_rank(smem_addr(ok ? &s_again : &s_abort), threadIdx.x)),
                   "r"(1)
                   : "memory");
    // nobody leaves while a copy of its own sums or into it may be under way
    hw_cluster_sync();
    ok = s_abort == 0;  // the same in every block of the cluster
    if (factors && s_again && ok) continue;
    if (ok)
      for (int j = threadIdx.x; j < nc; j += LS_THREADS)
        a.gpot[(size_t)b * a.N + c0 + j] = factors ? cap[j] : g[j];
    break;
  }
}

// The cluster for step l of B scenes of N: as many blocks as let all scenes
// run at once (at most 16, at most `wide` clusters of 16, 64 columns a block
// or more), then as many again as it takes for the rows to fit.  1024 tokens,
// 102 picks: 4.6 ms on 16 blocks, 5.6 on 8, 7.8 on 4.  False: the rows do not
// fit, and the step runs one launch a phase over the whole device (2500
// tokens: from 245 rows on; 375 picks 61 ms, 105 with every step so).
bool sink_shape(SinkArgs& a, int64_t B, int64_t N, int l, int wide, const DeviceInfo& di,
                size_t* smem) {
  const int cmax = wide > 0 ? 16 : 8;
  int c = cmax;
  while (c > 1 && (B * c > di.sm_count || N / c < 64 || (c == 16 && B > wide))) c >>= 1;
  for (; c <= cmax; c <<= 1) {
    a.CB = c;
    a.W = (int)(((N + c - 1) / c + 3) & ~(int64_t)3);
    a.pitch = ((a.W + 27) & ~31) + 4;  // 4 mod 32, at least W
    a.lp = ((l + 11) & ~15) + 4;       // 4 mod 16
    *smem = sizeof(float) * ((size_t)l * a.pitch + 2 * (size_t)a.W + (size_t)l) +
            sizeof(float2) * (size_t)(2 + 2 * c) * (size_t)a.lp;
    if (*smem + 1024 <= (size_t)di.max_smem_optin) return true;
  }
  return false;
}

// score(t) = sum_{j in M_g(t)} r_j C(t, j) for every unselected t; the
// block's smallest (score, index) key goes to keys[b][l] by atomicMin.
__global__ void __launch_bounds__(LIT_THREADS) k_lit_score(
    const float* __restrict__ C, int64_t ldc, int N, int K, int l, int g, int kk,
    const int32_t* __restrict__ nbr, const float* __restrict__ resid,
    const uint8_t* __restrict__ chosen, unsigned long long* __restrict__ keys) {
  __shared__ unsigned long long s_min[LIT_THREADS / 32];
  const int b = blockIdx.y;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = blockIdx.x * (LIT_THREADS / 32) + w;
  unsigned long long key = ~0ull;
  if (t < N && !chosen[(size_t)b * N + t]) {
    const float* row = C + ((size_t)b * N + t) * ldc;
    const float* r = resid + (size_t)b * N;
    float s = 0.0f;
    if (g >= N) {
      for (int j0 = lane; j0 - lane < N; j0 += 16 * 32) {
        float x[16], y[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          const int j = j0 + 32 * u;
          x[u] = j < N ? __ldg(r + j) : 0.0f;
          y[u] = j < N ? __ldg(row + j) : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < 16; ++u) s = fmaf(x[u], y[u], s);
      }
    } else {
      if (lane == 0) s = r[t] * row[t];
      const int32_t* nb = nbr + ((size_t)b * N + t) * kk;
      for (int q = lane; q < g - 1; q += 32) {
        const int jj = __ldg(nb + q);
        s = fmaf(__ldg(r + jj), __ldg(row + jj), s);
      }
    }
    s = warp_sum(s);
    s = s > 0.0f ? s : 0.0f;  // a -0 sum keys as +0
    key = ((unsigned long long)__float_as_uint(s) << 32) | (uint32_t)t;
  }
  key = warp_min_u64(key);
  if (lane == 0) s_min[w] = key;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long m = s_min[0];
    for (int i = 1; i < LIT_THREADS / 32; ++i) m = s_min[i] < m ? s_min[i] : m;
    if (m != ~0ull) atomicMin(keys + (size_t)b * K + l, m);
  }
}

// The K picks in order, their scores, and the coverage objective of the
// selected set, F(S) = sum_j v_j min(m0, min_{s in S, j in M_g(s)} C(s, j)),
// in double: thread r sums j = r, r + blockDim, ... in order, then a fixed
// tree over the block.  One block (1024 threads) per scene; m in shared
// memory (N floats), lowered with integer atomicMin on the bit patterns of
// the non-negative costs.
__global__ void __launch_bounds__(1024) k_lit_finish(
    const float* __restrict__ C, int64_t ldc, int N, int K, int g, int kk,
    const int32_t* __restrict__ nbr, const float* __restrict__ v,
    const unsigned long long* __restrict__ keys, float m0, int32_t* __restrict__ order32,
    float* __restrict__ gains, double* __restrict__ objective) {
  extern __shared__ float sm_m[];
  __shared__ double s_red[32];
  const int b = blockIdx.x;
  for (int l = threadIdx.x; l < K; l += blockDim.x) {
    const unsigned long long k = keys[(size_t)b * K + l];
    order32[(size_t)b * K + l] = key_index(k);
    if (gains) gains[(size_t)b * K + l] = __uint_as_float((uint32_t)(k >> 32));
  }
  if (!objective) return;
  for (int j = threadIdx.x; j < N; j += blockDim.x) sm_m[j] = m0;
  __syncthreads();
  const float* Cb = C + (size_t)b * N * ldc;
  unsigned int* mbits = reinterpret_cast<unsigned int*>(sm_m);
  for (int l = 0; l < K; ++l) {
    const int s = key_index(keys[(size_t)b * K + l]);
    const float* row = Cb + (size_t)s * ldc;
    if (g >= N) {
      for (int j = threadIdx.x; j < N; j += blockDim.x) {
        const float c = __ldg(row + j);
        atomicMin(mbits + j, __float_as_uint(c > 0.0f ? c : 0.0f));  // -0 as +0
      }
    } else {
      for (int q = threadIdx.x; q < g; q += blockDim.x) {
        const int j = q == 0 ? s : __ldg(nbr + ((size_t)b * N + s) * kk + q - 1);
        const float c = __ldg(row + j);
        atomicMin(mbits + j, __float_as_uint(c > 0.0f ? c : 0.0f));
      }
    }
  }
  __syncthreads();
  double acc = 0.0;
  for (int j = threadIdx.x; j < N; j += blockDim.x)
    acc += (double)v[(size_t)b * N + j] * (double)sm_m[j];
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double F = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) F += s_red[i];
    objective[b] = F;
  }
}

// k_lit_sinkhorn's launch; *wide: how many clusters of 16 with all of a
// block's shared memory the device holds at once.
int sink_config(const DeviceInfo& di, cudaStream_t s, cudaLaunchConfig_t* cfg,
                cudaLaunchAttribute* attr, int* wide) {
  CP_TRY_STATUS(cuda_status(
      cudaFuncSetAttribute(k_lit_sinkhorn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           di.max_smem_optin - 1024),
      "launch_sgs_literal: smem attribute"));
  cfg->gridDim = dim3(16);
  cfg->blockDim = dim3(LS_THREADS);
  cfg->dynamicSmemBytes = (size_t)di.max_smem_optin - 1024;
  cfg->stream = s;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = 16;
  attr->val.clusterDim.y = 1;
  attr->val.clusterDim.z = 1;
  cfg->attrs = attr;
  cfg->numAttrs = 1;
  *wide = 0;
  if (cudaFuncSetAttribute(k_lit_sinkhorn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveClusters(wide, (const void*)k_lit_sinkhorn, cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    *wide = 0;
  }
  return CP_OK;
}

}  // namespace

size_t sgs_literal_ws_bytes(int64_t B, int64_t N, int64_t K) {
  auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
  const size_t BN = (size_t)B * (size_t)N, BK = (size_t)B * (size_t)K;
  return up(sizeof(float) * BK) + up(sizeof(float) * BN) + up(sizeof(float) * BN) +
         up(sizeof(unsigned long long) * BK) + up(BN);
}

int launch_sgs_literal(const float* cost, int64_t ldc, const int32_t* nbr, const float* v,
                       const DevParams& P, int64_t B, int64_t N, int64_t K, int32_t* order32,
                       float* gains, double* objective, void* scratch, int* status, cudaStream_t s) {
  if (B <= 0 || N <= 0 || K <= 0) return CP_OK;
  auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
  const size_t BN = (size_t)B * (size_t)N, BK = (size_t)B * (size_t)K;
  unsigned char* base = static_cast<unsigned char*>(scratch);
  float* fpot = reinterpret_cast<float*>(base);
  float* gpot = reinterpret_cast<float*>(base + up(sizeof(float) * BK));
  float* resid = reinterpret_cast<float*>(base + up(sizeof(float) * BK) + up(sizeof(float) * BN));
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(
      base + up(sizeof(float) * BK) + 2 * up(sizeof(float) * BN));
  uint8_t* chosen = base + up(sizeof(float) * BK) + 2 * up(sizeof(float) * BN) +
                    up(sizeof(unsigned long long) * BK);
  CP_TRY_STATUS(cuda_status(cudaMemsetAsync(keys, 0xFF, sizeof(unsigned long long) * BK, s),
                            "launch_sgs_literal: keys"));
  CP_TRY_STATUS(cuda_status(cudaMemsetAsync(gpot, 0, sizeof(float) * BN, s),
                            "launch_sgs_literal: potentials"));
  CP_TRY_STATUS(cuda_status(cudaMemsetAsync(chosen, 0, BN, s), "launch_sgs_literal: chosen"));
  const float eps = P.sot_eps, inv_eps = 1.0f / P.sot_eps;
  const float log_u = (float)(-log((double)K));
  const int n = (int)N, k = (int)K, g = P.g, kk = P.kk;
  const dim3 gcols((unsigned)((N + LC_COLS - 1) / LC_COLS), (unsigned)B);
  const dim3 bcols(LC_COLS, LC_GROUPS);
  const dim3 gscore((unsigned)((N + LIT_THREADS / 32 - 1) / (LIT_THREADS / 32)), (unsigned)B);
  DeviceInfo di;
  if (device_info(&di) != CP_OK) return CP_ECUDA;
  SinkArgs sa{cost, keys, v, gpot, resid, chosen, ldc, n, k, 0, P.sot_iters,
              0,    0,    0, 0, eps, inv_eps,
              (float)(1.0 / (double)eps - (double)inv_eps), (float)(1.4426950408889634 / (double)eps),
              eps * log_u, (float)(1.0 / (double)K), status, P.timeout_ns};
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[1];
  int wide = 0;
  CP_TRY_STATUS(sink_config(di, s, &cfg, attr, &wide));
  for (int l = 0; l < k; ++l) {
    size_t sink_smem = 0;
    if (l > 0 && sink_shape(sa, B, N, l, wide, di, &sink_smem)) {
      sa.l = l;
      attr->val.clusterDim.x = (unsigned)sa.CB;
      cfg.gridDim = dim3((unsigned)(B * sa.CB));
      cfg.dynamicSmemBytes = sink_smem;
      const cudaError_t e = cudaLaunchKernelEx(&cfg, k_lit_sinkhorn, sa);
      note_launch();
      CP_TRY_STATUS(cuda_status(e, "launch_sgs_literal: iterations"));
      k_lit_score<<<gscore, LIT_THREADS, 0, s>>>(cost, ldc, n, k, l, g, kk, nbr, resid, chosen,
                                                 keys);
      CP_TRY_STATUS(last_launch_status());
      continue;
    }
    if (l > 0) {
      const dim3 grows((unsigned)l, (unsigned)B);
      for (int it = 0; it < P.sot_iters; ++it) {
        k_lit_rows<<<grows, LIT_THREADS, 0, s>>>(cost, ldc, n, k, l, keys, gpot, eps, inv_eps,
                                                 log_u, fpot);
        CP_TRY_STATUS(last_launch_status());
        k_lit_cols<false><<<gcols, bcols, 0, s>>>(cost, ldc, n, k, l, keys, fpot, v, eps,
                                                  inv_eps, gpot, resid, chosen);
        CP_TRY_STATUS(last_launch_status());
      }
    }
    k_lit_cols<true><<<gcols, bcols, 0, s>>>(cost, ldc, n, k, l, keys, fpot, v, eps, inv_eps,
                                             gpot, resid, chosen);
    CP_TRY_STATUS(last_launch_status());
    k_lit_score<<<gscore, LIT_THREADS, 0, s>>>(cost, ldc, n, k, l, g, kk, nbr, resid, chosen,
                                               keys);
    CP_TRY_STATUS(last_launch_status());
  }
  const size_t smem = sizeof(float) * (size_t)N;
  CP_TRY_STATUS(allow_smem((const void*)k_lit_finish, smem, "launch_sgs_literal: smem attribute"));
  k_lit_finish<<<(unsigned)B, 1024, smem, s>>>(cost, ldc, n, k, g, kk, nbr, v, keys, P.m0,
                                               order32, gains, objective);
  return last_launch_status();
}

}  // namespace cp
