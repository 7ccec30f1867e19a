// K5: Spatial-Guided Greedy Selection (Sec. 3.5, Eqs. srpot, local_neighbor,
// greedy_flow, sgs_select, sgs_update), every gain every step (sgs_mode 1; the
// default selection of a few tokens, behind bounds), and the choice between the
// selection kernels (sgs_push.cu holds the default one, sgs_literal.cu the rule
// as printed).
//
// The semi-relaxed OT of Eq. srpot, with the source support and its capacity
// as decision variables, has a closed-form plan: every target t_j sends its
// mass v_j to its cheapest selected source among those whose neighbourhood
// M_g contains it.  Its value is F(S) = sum_j v_j m_j with the coverage cost
// m_j = min(m0, min_{s in S, j in M_g(s)} C(s, j)), and the residual-weighted
// marginal cost of adding t is -gain(t) with
//     gain(t) = sum_{j in M_g(t)} v_j max(m_j - C(t, j), 0).
// Each step adds the unselected token with the largest gain (lowest index
// among equal gains) and lowers m on its neighbourhood.
//
// One persistent cooperative grid: each scene owns `cps` co-resident blocks.
// Every block keeps the whole (m_j, v_j) state of its scene in shared memory;
// per step the blocks sweep disjoint candidate rows (one warp per row,
// float4 streaming loads of C), publish their best (gain, index) key, meet at
// a scene-local grid barrier (bounded wait), all reduce the same partials to
// the same winner and apply the same update to their copy of m.
#include <math.h>

#include "sgs_gain.cuh"

namespace cp {

constexpr int SGS_THREADS = 512;
constexpr int SGS_WARPS = SGS_THREADS / 32;

// fx of fixed_term: S = 190 - fx = 60 - floor(log2 m0) keeps a gain (at most
// m0 up to rounding) below 2^62; not below 64, so that a zero term stays 0
// (m0 below 2^-66 then loses resolution under 2^-126).
int gain_fx(float m0) {
  if (!(m0 > 0.0f)) return 64;
  const int e = isfinite(m0) ? ilogbf(m0) : 128;
  return 130 + e < 64 ? 64 : 130 + e;
}

// A cost is at most the sum of its weights, up to rounding (which the scale's
// spare bit takes).
int gain_fx_covered(const DevParams& P) {
  const float c = P.lambda_f + P.lambda_x + P.lambda_tau;
  return gain_fx(c < P.m0 ? c : P.m0);
}

// FEW (dense): the default selection of few tokens, its first pick given.  A
// gain computed at an earlier step bounds the current one, so a candidate
// whose bound is not above the best gain that any warp of the scene has found
// in this step is passed over; each warp evaluates its highest bound first.
struct FewArgs {
  const gain_t* first;          // [B] key of the first pick
  float* bound;                 // [B][N] at the start: sums of the first gains, inexact
  unsigned long long* running;  // [B][2] zeros: the best key so far, by turn
};
template <bool LOCAL, bool FEW>
__global__ void __launch_bounds__(SGS_THREADS, LOCAL ? 3 : 2) k_sgs(
    const float* __restrict__ cost, int64_t ldc, const float* __restrict__ slab,
    const int32_t* __restrict__ nbr, const float* __restrict__ v_all, DevParams P, int N, int K,
    int cps, int scene0, int fx, int fx1, FewArgs few, int32_t* __restrict__ order32,
    float* __restrict__ gains, double* __restrict__ objective, unsigned long long* partials,
    uint32_t* counters, int* status) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int ncols = LOCAL ? N : (int)ldc;  // dense rows are padded to ldc (C = 0, v = 0)
  float* sm_m = reinterpret_cast<float*>(smem);                  // [ncols] coverage cost m_j
  float* sm_v = sm_m + ncols;                                    // [ncols] capacity v_j
  uint32_t* chosen = reinterpret_cast<uint32_t*>(sm_v + ncols);  // [ceil(N/32)] bitset
  __shared__ unsigned long long s_best[SGS_WARPS];
  __shared__ int s_pick, s_bad, s_fx;
  __shared__ float s_gain;

  const int b = scene0 + blockIdx.x / cps;
  const int c = blockIdx.x % cps;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float* v = v_all + (size_t)b * N;
  const float* Cb = LOCAL ? nullptr : cost + (size_t)b * N * ldc;
  const float* Sb = LOCAL ? slab + (size_t)b * N * P.g : nullptr;
  const int32_t* NB = nbr + (size_t)b * N * P.kk;
  unsigned long long* part = partials;  // [2][B][cps]
  const int nchosen = (N + 31) >> 5;

  for (int j = threadIdx.x; j < ncols; j += SGS_THREADS) {
    sm_m[j] = j < N ? P.m0 : 0.0f;
    sm_v[j] = j < N ? v[j] : 0.0f;
  }
  for (int i = threadIdx.x; i < nchosen; i += SGS_THREADS) chosen[i] = 0u;
  __syncthreads();
  // the scale after the first pick: m0's while a target is still uncovered (its
  // cost undefined, as of a token with an infinite coordinate)
  auto second_scale = [&]() -> int {
    if (fx1 == fx) return fx;
    bool open = false;
    for (int j = threadIdx.x; j < N; j += SGS_THREADS) open |= !(sm_m[j] < P.m0);
    return __syncthreads_or(open) ? fx : fx1;
  };
  int step = 0;
  if (FEW) {  // the first pick is known
    const gain_t key = few.first[b];
    const int pick = key_token(key);
    for (int j = threadIdx.x; j < N; j += SGS_THREADS)
      sm_m[j] = fminf(sm_m[j], __ldg(Cb + (size_t)pick * ldc + j));
    if (threadIdx.x == 0) {
      chosen[pick >> 5] = 1u << (pick & 31);
      if (c == 0) {
        order32[(size_t)b * K] = pick;
        if (gains) gains[(size_t)b * K] = key_gain(key);
      }
    }
    step = 1;
    __syncthreads();
    fx = second_scale();
  }

  const int gw = c * SGS_WARPS + w, nw = cps * SGS_WARPS;
  const size_t nscenes = gridDim.x / cps;
  bool alive = true;
  unsigned long long my_evals = 0ull;  // rows this warp evaluated (lane 0 counts)
  unsigned long long my_update_bytes = 0ull;  // coverage-update reads (thread 0 of block 0)
  uint32_t turn = 0;  // sweeps: one a step, one more where the scale is refitted
  while (step < K && alive) {
    unsigned long long best = 0ull;
    if (FEW) {
      float* bound = few.bound + (size_t)b * N;
      // this turn's slot; the other's last readers are behind the last barrier
      unsigned long long* run = few.running + 2 * (size_t)b;
      if (c == 0 && threadIdx.x == 0) run[(turn + 1u) & 1u] = 0ull;
      run += turn & 1u;
      // what the gain of candidate i of this warp is known not to exceed
      auto above = [&](int i) -> gain_t {
        const int t = gw + i * nw;
        if (t >= N || (chosen[t >> 5] & (1u << (t & 31)))) return 0ull;
        // 1 + 2^-15: the first sums are as far off (k_first_bounds)
        const float x = __fmul_ru(__ldcg(bound + t), 1.000030517578125f);
        return gain_key(__float_as_uint(x), t);
      };
      auto evaluate = [&](int t) {
        const gain_t acc = dense_row_gain(Cb + (size_t)t * ldc, sm_m, sm_v, ncols, fx, lane);
        ++my_evals;
        const uint32_t bits = gain_bits(acc, fx);
        const gain_t key = gain_key(bits, t);
        if (lane == 0) {
          __stcg(bound + t, __uint_as_float(bits));
          if (key > best) atomicMax(run, key);
        }
        best = key > best ? key : best;
      };
      const int mine = gw < N ? (N - gw + nw - 1) / nw : 0;
      gain_t top = 0ull;
      for (int i = lane; i < mine; i += 32) top = max(top, above(i));
      top = warp_max_key(top);
      const int seed = top ? key_token(top) : -1;
      if (seed >= 0) evaluate(seed);
      for (int i0 = 0; i0 < mine; i0 += 32) {
        const gain_t k = i0 + lane < mine ? above(i0 + lane) : 0ull;
        uint32_t todo = 0xFFFFFFFFu;
        while (todo) {
          const gain_t seen = warp_max_key(lane == 0 ? *(volatile gain_t*)run : best);
          todo &= __ballot_sync(0xFFFFFFFFu, k > seen && gw + (i0 + lane) * nw != seed);
          if (!todo) break;
          const int l = __ffs(todo) - 1;
          todo &= todo - 1u;
          evaluate(gw + (i0 + l) * nw);
        }
      }
    } else {
      for (int t = gw; t < N; t += nw) {
        if (chosen[t >> 5] & (1u << (t & 31))) continue;
        const gain_t acc =
            LOCAL ? local_row_gain(Sb + (size_t)t * P.g, NB + (size_t)t * P.kk, t, P.g, sm_m, sm_v,
                                   fx, lane)
                  : dense_row_gain(Cb + (size_t)t * ldc, sm_m, sm_v, ncols, fx, lane);
        ++my_evals;
        const unsigned long long key = gain_key(gain_bits(acc, fx), t);
        best = key > best ? key : best;
      }
    }
    if (lane == 0) s_best[w] = best;
    __syncthreads();
    const int par = (int)(turn & 1u);
    ++turn;
    if (threadIdx.x == 0) {
      unsigned long long m = s_best[0];
      for (int i = 1; i < SGS_WARPS; ++i) m = s_best[i] > m ? s_best[i] : m;
      part[((size_t)par * nscenes + (b - scene0)) * cps + c] = m;
    }
    if (!grid_barrier(counters + b, turn * (uint32_t)cps, status, P.timeout_ns)) {
      alive = false;
      break;
    }
    if (w == 0) {
      unsigned long long m = 0ull;
      const unsigned long long* pp = part + ((size_t)par * nscenes + (b - scene0)) * cps;
      for (int i = lane; i < cps; i += 32) {
        // each reading lane acquires: a weak load may be served a stale copy
        const unsigned long long x = ld_acquire_u64(pp + i);
        m = x > m ? x : m;
      }
      m = warp_max_u64(m);
      if (lane == 0) {
        const int pk = key_token(m);
        s_pick = pk;
        s_gain = key_gain(m);
        // decided once, before anyone updates the state: a winner must be an
        // unselected token (never expected to fail)
        s_fx = fx;
        if (m != 0ull && (LOCAL || step > 0) && (uint32_t)(m >> 32) <= gain_floor(fx))
          s_fx = gain_refit((uint32_t)(m >> 32) - 1u, fx, 32 - __clz(N));
        s_bad = m == 0ull || pk < 0 || pk >= N || (chosen[pk >> 5] & (1u << (pk & 31))) != 0u;
      }
    }
    __syncthreads();
    const int pick = s_pick;
    if (s_bad) {
      if (threadIdx.x == 0 && atomicCAS(status, 0, CP_EDEVICE) == 0) {
        status[4] = step;  // where it happened, for diagnosis
        status[5] = b;
        status[6] = c;
        status[7] = pick;
      }
      alive = false;
      break;
    }
    if (s_fx != fx) {  // every block's answer is the same
      fx = s_fx;
      // the bounds are of sums cut at the scale before
      if (FEW)
        for (int t = gw + lane * nw; t < N; t += 32 * nw)
          __stcg(few.bound + (size_t)b * N + t, 1.0e38f);
      __syncthreads();  // before it is written again
      continue;
    }
    if (threadIdx.x == 0) {
      chosen[pick >> 5] |= 1u << (pick & 31);
      if (c == 0) {
        order32[(size_t)b * K + step] = pick;
        if (gains) gains[(size_t)b * K + step] = s_gain;
        my_update_bytes += LOCAL ? 8ull * (unsigned long long)P.g : 4ull * (unsigned long long)N;
      }
    }
    // S <- S u {t*} (Eq. sgs_update): lower the coverage cost of its targets
    if (!LOCAL) {
      const float* row = Cb + (size_t)pick * ldc;
      for (int j = threadIdx.x; j < N; j += SGS_THREADS) sm_m[j] = fminf(sm_m[j], __ldg(row + j));
    } else {
      const float* srow = Sb + (size_t)pick * P.g;
      const int32_t* nb = NB + (size_t)pick * P.kk;
      for (int k = threadIdx.x; k < P.g; k += SGS_THREADS) {
        const int j = k == 0 ? pick : nb[k - 1];
        sm_m[j] = fminf(sm_m[j], srow[k]);
      }
    }
    __syncthreads();
    if (++step == 1) fx = second_scale();
  }

  unsigned long long* cstats = reinterpret_cast<unsigned long long*>(
      reinterpret_cast<unsigned char*>(status) + kCallStatsOffset);
  if (lane == 0 && my_evals) atomicAdd(&cstats[0], my_evals);
  if (c == 0 && threadIdx.x == 0) atomicAdd(&cstats[1], (unsigned long long)K);
  if (lane == 0 && my_evals)
    atomicAdd(&cstats[2], my_evals * (unsigned long long)(LOCAL ? 8 * P.g : 4 * ldc));
  if (my_update_bytes) atomicAdd(&cstats[2], my_update_bytes);
  if (c == 0 && alive && objective) {
    const double F = objective_sum(sm_m, sm_v, N);
    if (threadIdx.x == 0) objective[b] = F;
  }
}

template <bool LOCAL, bool FEW>
static int sgs_launch_impl(const float* cost, int64_t ldc, const float* slab, const int32_t* nbr,
                           const float* v, const DevParams& P, int64_t B, int64_t N, int64_t K,
                           int32_t* order32, float* gains, double* objective,
                           unsigned long long* partials, uint32_t* counters, int* status,
                           cudaStream_t s, FewArgs few = FewArgs{}) {
  DeviceInfo di;
  if (device_info(&di) != CP_OK) return CP_ECUDA;
  const int64_t ncols = LOCAL ? N : ldc;
  const size_t smem = 2 * sizeof(float) * (size_t)ncols + sizeof(uint32_t) * (size_t)((N + 31) / 32);
  auto fn = k_sgs<LOCAL, FEW>;
  CP_TRY_STATUS(allow_smem((const void*)fn, smem, "launch_sgs: smem attribute"));
  int per_sm = 0;
  if (cuda_status(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, SGS_THREADS, smem),
                  "launch_sgs: occupancy") != CP_OK)
    return CP_ECUDA;
  if (per_sm < 1) return CP_EUNSUPPORTED;
  const int64_t slots = (int64_t)per_sm * di.sm_count;
  const int64_t per_launch = B < slots ? B : slots;  // scenes resident together
  int cps = (int)(slots / per_launch);
  // a scene never needs more blocks than it has candidate rows per warp
  const int64_t max_cps = (N + SGS_WARPS - 1) / SGS_WARPS;
  if (cps > max_cps) cps = (int)max_cps;
  if (cps < 1) cps = 1;
  if (cuda_status(cudaMemsetAsync(counters, 0, sizeof(uint32_t) * (size_t)B, s),
                  "launch_sgs: counters") != CP_OK)
    return CP_ECUDA;
  if (cuda_status(cudaMemsetAsync(partials, 0,
                                  sizeof(unsigned long long) * 2 * (size_t)per_launch * cps, s),
                  "launch_sgs: partials") != CP_OK)
    return CP_ECUDA;
  for (int64_t b0 = 0; b0 < B; b0 += per_launch) {
    const int64_t nb = (B - b0) < per_launch ? (B - b0) : per_launch;
    int Ni = (int)N, Ki = (int)K, scene0 = (int)b0, fx = gain_fx(P.m0);
    int fx1 = LOCAL ? fx : gain_fx_covered(P);  // from the second step on
    DevParams Pc = P;
    void* args[] = {(void*)&cost, (void*)&ldc, (void*)&slab, (void*)&nbr, (void*)&v, (void*)&Pc,
                    (void*)&Ni, (void*)&Ki, (void*)&cps, (void*)&scene0, (void*)&fx, (void*)&fx1,
                    (void*)&few, (void*)&order32, (void*)&gains, (void*)&objective,
                    (void*)&partials, (void*)&counters, (void*)&status};
    cudaError_t e = cudaLaunchCooperativeKernel((const void*)fn, dim3((unsigned)(nb * cps)),
                                                dim3(SGS_THREADS), args, smem, s);
    note_launch();
    if (cuda_status(e, "launch_sgs: cooperative launch") != CP_OK) return CP_ECUDA;
  }
  return CP_OK;
}

int launch_sgs(const float* cost, int64_t ldc, const float* slab, const int32_t* nbr,
               const float* v, const DevParams& P, int64_t B, int64_t N, int64_t K,
               int32_t* order32, float* gains, double* objective, uint64_t* partials,
               uint32_t* counters, int* status, cudaStream_t s, const float* g0, void* push_ws,
               int64_t push_wave) {
  auto* part = reinterpret_cast<unsigned long long*>(partials);
  if (few_picks(P, N, K)) {
    FewArgs few;
    CP_TRY_STATUS(launch_first_pick(cost, ldc, v, P, B, N, s, g0, push_ws, &few.first, &few.bound,
                                    &few.running));
    return sgs_launch_impl<false, true>(cost, ldc, slab, nbr, v, P, B, N, K, order32, gains,
                                        objective, part, counters, status, s, few);
  }
  if (P.sgs_mode == 0)
    return launch_sgs_push(cost, ldc, slab, nbr, v, P, B, N, K, order32, gains, objective, status,
                           s, g0, push_ws, push_wave);
  if (P.g < N)
    return sgs_launch_impl<true, false>(cost, ldc, slab, nbr, v, P, B, N, K, order32, gains,
                                        objective, part, counters, status, s);
  return sgs_launch_impl<false, false>(cost, ldc, slab, nbr, v, P, B, N, K, order32, gains,
                                       objective, part, counters, status, s);
}

// Upper bound of the partial slots the launcher may use: 2 * B * cps with
// cps <= ceil(N / SGS_WARPS).
int64_t sgs_partials_count(int64_t B, int64_t N) {
  return 2 * B * ((N + SGS_WARPS - 1) / SGS_WARPS);
}

// ---------------------------------------------------------------------------
// Barrier self-test: n_blocks co-resident blocks wait for `expected`
// arrivals; with expected > n_blocks the bounded wait must run out.
// ---------------------------------------------------------------------------
__global__ void k_barrier_selftest(uint32_t* ctr, uint32_t expected, int* status,
                                   uint64_t timeout_ns) {
  grid_barrier(ctr, expected, status, timeout_ns);
}

int launch_barrier_selftest(int n_blocks, int expected, uint64_t timeout_ns, uint32_t* ctr,
                            int* status, cudaStream_t s) {
  DeviceInfo di;
  if (device_info(&di) != CP_OK) return CP_ECUDA;
  if (n_blocks < 1 || n_blocks > di.sm_count || expected < 0) return CP_EINVAL;
  if (cudaMemsetAsync(ctr, 0, sizeof(uint32_t), s) != cudaSuccess) return CP_ECUDA;
  if (cudaMemsetAsync(status, 0, sizeof(int), s) != cudaSuccess) return CP_ECUDA;
  uint32_t exp_u = (uint32_t)expected;
  void* args[] = {(void*)&ctr, (void*)&exp_u, (void*)&status, (void*)&timeout_ns};
  cudaError_t e = cudaLaunchCooperativeKernel((const void*)k_barrier_selftest, dim3(n_blocks),
                                              dim3(64), args, 0, s);
  note_launch();
  return cuda_status(e);
}

// ---------------------------------------------------------------------------
// Ascending sort of K indices per scene (bitonic, shared memory).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(1024) k_sort_kept(const int32_t* __restrict__ idx32, int K, int L,
                                                    int64_t* __restrict__ kept,
                                                    int64_t* __restrict__ order64) {
  extern __shared__ int32_t sk[];
  const int b = blockIdx.x;
  const int32_t* in = idx32 + (size_t)b * K;
  for (int i = threadIdx.x; i < L; i += blockDim.x) sk[i] = i < K ? in[i] : INT32_MAX;
  if (order64)
    for (int i = threadIdx.x; i < K; i += blockDim.x) order64[(size_t)b * K + i] = in[i];
  __syncthreads();
  for (int size = 2; size <= L; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int i = threadIdx.x; i < (L >> 1); i += blockDim.x) {
        const int a = 2 * i - (i & (stride - 1));
        const int c = a + stride;
        const bool up = (a & size) == 0;
        const int32_t x = sk[a], y = sk[c];
        if ((x > y) == up) { sk[a] = y; sk[c] = x; }
      }
      __syncthreads();
    }
  }
  for (int i = threadIdx.x; i < K; i += blockDim.x) kept[(size_t)b * K + i] = sk[i];
}

int launch_sort_kept(const int32_t* idx32, int64_t B, int64_t K, int64_t* kept, int64_t* order64,
                     cudaStream_t s) {
  int L = 2;
  while (L < K) L <<= 1;
  const size_t smem = sizeof(int32_t) * (size_t)L;
  CP_TRY_STATUS(allow_smem((const void*)k_sort_kept, smem, "launch_sort_kept: smem attribute"));
  k_sort_kept<<<(unsigned)B, 1024, smem, s>>>(idx32, (int)K, L, kept, order64);
  return last_launch_status();
}

}  // namespace cp
