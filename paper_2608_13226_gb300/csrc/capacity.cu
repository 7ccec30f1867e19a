// K4: FST capacity (Sec. 3.4, Eqs. fst_capacity_score, fst_capacity) and the
// cost slab of the local SGS neighbourhoods (Eq. local_neighbor).
#include "common.cuh"
#include "bf16_dot.cuh"

namespace cp {

// r_j = (1/n) sum_{k in N_n(j)} alpha_f d^_f(j,k) + alpha_x d^_x(j,k) + alpha_tau d^_tau(j,k)
// One block per token, one warp per neighbour (warp w takes k = N_n(j)[q]
// for q = w, w + warps, ...): the warps read the token's own row together,
// so L1 serves it once for all of them, and each reads one neighbour row.
// The dot products run over 16-byte feature vectors; the terms are summed in
// neighbour order by one thread.
constexpr int CAP_WARPS = 8;

template <typename T>
__device__ __forceinline__ float row_dot(const T* a, const T* b, int D, int lane) {
  constexpr int V = Vec16<T>::n;
  float dot = 0.0f;
  for (int d = lane * V; d < D; d += 32 * V) {
    float x[V], y[V];
    Vec16<T>::load(a + d, x);
    Vec16<T>::load(b + d, y);
#pragma unroll
    for (int i = 0; i < V; ++i) dot = fmaf(x[i], y[i], dot);
  }
  return dot;
}
template <>
__device__ __forceinline__ float row_dot<__nv_bfloat16>(const __nv_bfloat16* a,
                                                        const __nv_bfloat16* b, int D, int lane) {
  float dot = 0.0f;
  for (int d = lane * 8; d < D; d += 256)
    dot = dot8_bf16(__ldg(reinterpret_cast<const uint4*>(a + d)),
                    __ldg(reinterpret_cast<const uint4*>(b + d)), dot);
  return dot;
}

template <typename T>
__global__ void __launch_bounds__(32 * CAP_WARPS) k_capacity_r(
    const T* __restrict__ F_all, const float* __restrict__ inv_all, const float* __restrict__ pos_all,
    const int32_t* __restrict__ frame_all, const SceneNorms* __restrict__ norms,
    const int32_t* __restrict__ nbr_all, DevParams P, int N, int D, float* __restrict__ r_all) {
  constexpr int CHUNK = 256;
  __shared__ float s_term[CHUNK];  // the terms of neighbours q0 .. q0 + CHUNK - 1
  const int j = blockIdx.x;
  const int b = blockIdx.y;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nw = (int)(blockDim.x >> 5);
  const T* F = F_all + (size_t)b * N * D;
  const float* inv = inv_all + (size_t)b * N;
  const float* X = pos_all + (size_t)b * N * 3;
  const int32_t* TAU = frame_all + (size_t)b * N;
  const int32_t* nb = nbr_all + ((size_t)b * N + j) * P.kk;
  const SceneNorms nm = norms[b];
  const T* fj = F + (size_t)j * D;
  float acc = 0.0f;  // thread 0's running sum, in neighbour order
  for (int q0 = 0; q0 < P.n_cap; q0 += CHUNK) {
    const int qn = min(CHUNK, P.n_cap - q0);
    for (int qq = w; qq < qn; qq += nw) {
      const int k = __ldg(nb + q0 + qq);
      const T* fk = F + (size_t)k * D;
      const float dot = warp_sum(row_dot<T>(fj, fk, D, lane));
      const float cosv = clamp_cos(dot * inv[j] * inv[k]);
      const float tf = ((1.0f - cosv) - nm.f_lo) * nm.f_rinv;
      const float dx = sqrtf(sqdist_rn(X[3 * j], X[3 * j + 1], X[3 * j + 2], X[3 * k],
                                       X[3 * k + 1], X[3 * k + 2]));
      const float tx = (dx - nm.x_lo) * nm.x_rinv;
      const int dt = TAU[j] - TAU[k];
      const float tt = dt > 0 ? (float)dt * nm.t_rinv : 0.0f;
      if (lane == 0) s_term[qq] = P.alpha_f * tf + P.alpha_x * tx + P.alpha_tau * tt;
    }
    __syncthreads();
    if (threadIdx.x == 0)
      for (int qq = 0; qq < qn; ++qq) acc += s_term[qq];
    __syncthreads();
  }
  if (threadIdx.x == 0) r_all[(size_t)b * N + j] = P.n_cap > 0 ? acc / (float)P.n_cap : 0.0f;
}

// The same r_j for bf16 features, a warp a token: its row against R of its
// neighbours' at a time.  A block's 8 tokens are neighbours themselves (their
// places follow the neighbour grid's order), so at any moment its warps read
// the same columns of few distinct rows, most of them from L1; a block a
// token, a warp a neighbour, brought every row from L2 each time it was a
// neighbour.  32 scenes of 8192, D = 3584, 8 neighbours: 15 GB of such rows,
// 1.31 ms, now 1.00; one scene of 16384 87 us, now 74.  Three blocks an SM:
// at the registers the compiler takes by itself one fits, and 1.99 ms.  Every
// dot product and sum keeps its order.
template <int R>
__global__ void __launch_bounds__(256, 3) k_capacity_r_near(
    const __nv_bfloat16* __restrict__ F_all, const float* __restrict__ inv_all,
    const float* __restrict__ pos_all, const int32_t* __restrict__ frame_all,
    const SceneNorms* __restrict__ norms, const int32_t* __restrict__ nbr_all,
    const float4* __restrict__ order_all, DevParams P, int N, int D, float* __restrict__ r_all) {
  const int slot = blockIdx.x * 8 + (threadIdx.x >> 5), b = blockIdx.y, lane = threadIdx.x & 31;
  if (slot >= N) return;
  const int j = __float_as_int(order_all[(size_t)b * N + slot].w);
  const __nv_bfloat16* F = F_all + (size_t)b * N * D;
  const float* inv = inv_all + (size_t)b * N;
  const float* X = pos_all + (size_t)b * N * 3;
  const int32_t* TAU = frame_all + (size_t)b * N;
  const int32_t* nb = nbr_all + ((size_t)b * N + j) * P.kk;
  const SceneNorms nm = norms[b];
  const __nv_bfloat16* fj = F + (size_t)j * D;
  float acc = 0.0f;
  for (int q0 = 0; q0 < P.n_cap; q0 += R) {
    const int mine = nb[min(q0 + (lane & (R - 1)), P.n_cap - 1)];
    const __nv_bfloat16* fk[R];
    float dot[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      fk[i] = F + (size_t)__shfl_sync(0xFFFFFFFFu, mine, i) * D;
      dot[i] = 0.0f;
    }
    for (int c = lane * 8; c < D; c += 256) {
      const uint4 x = __ldg(reinterpret_cast<const uint4*>(fj + c));
      uint4 y[R];
#pragma unroll
      for (int i = 0; i < R; ++i) y[i] = __ldg(reinterpret_cast<const uint4*>(fk[i] + c));
#pragma unroll
      for (int i = 0; i < R; ++i) dot[i] = dot8_bf16(x, y[i], dot[i]);
    }
    float own = 0.0f;
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const float t = warp_sum(dot[i]);
      own = (lane & (R - 1)) == i ? t : own;
    }
    const int k = mine;
    const float cosv = clamp_cos(own * inv[j] * inv[k]);
    const float tf = ((1.0f - cosv) - nm.f_lo) * nm.f_rinv;
    const float dx = sqrtf(
        sqdist_rn(X[3 * j], X[3 * j + 1], X[3 * j + 2], X[3 * k], X[3 * k + 1], X[3 * k + 2]));
    const float tx = (dx - nm.x_lo) * nm.x_rinv;
    const int dt = TAU[j] - TAU[k];
    const float tt = dt > 0 ? (float)dt * nm.t_rinv : 0.0f;
    const float term = P.alpha_f * tf + P.alpha_x * tx + P.alpha_tau * tt;
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const float t = __shfl_sync(0xFFFFFFFFu, term, i);
      if (q0 + i < P.n_cap) acc += t;
    }
  }
  if (lane == 0) r_all[(size_t)b * N + j] = P.n_cap > 0 ? acc / (float)P.n_cap : 0.0f;
}

// The same r_j from stored cosines in place of the dot product, the rest
// identical: the normaliser Gram's output, the upper triangle of
// [B][N][ldc] (cos(j, k) at [min(j, k)][max(j, k)]); or, given pos_of, the
// flagged Morton tiles of the local path (cos(j, k) at [min(pos)][max(pos)]).
// One thread per token; its n gathers fall in one row, near its own index
// (nearest neighbours sit in the same or adjacent frames).
__global__ void __launch_bounds__(256) k_capacity_r_cos(
    const float* __restrict__ cos_all, int64_t ldc, const float* __restrict__ pos_all,
    const int32_t* __restrict__ frame_all, const SceneNorms* __restrict__ norms,
    const int32_t* __restrict__ nbr_all, DevParams P, int N, const int32_t* __restrict__ pos_of,
    float* __restrict__ r_all) {
  const int j = blockIdx.x * 256 + threadIdx.x;
  const int b = blockIdx.y;
  if (j >= N) return;
  const int32_t* po = pos_of ? pos_of + (size_t)b * N : nullptr;
  const float* crow = cos_all + ((size_t)b * N + j) * (size_t)ldc;
  const float* X = pos_all + (size_t)b * N * 3;
  const int32_t* TAU = frame_all + (size_t)b * N;
  const int32_t* nb = nbr_all + ((size_t)b * N + j) * P.kk;
  const SceneNorms nm = norms[b];
  const float xj = X[3 * j], yj = X[3 * j + 1], zj = X[3 * j + 2];
  const int tj = TAU[j];
  float acc = 0.0f;
  for (int q = 0; q < P.n_cap; ++q) {
    const int k = nb[q];
    float cosv;
    if (po) {
      const int a = po[j], c = po[k];
      cosv = cos_all[((size_t)b * N + min(a, c)) * (size_t)ldc + max(a, c)];
    } else {
      cosv = k > j ? crow[k] : cos_all[((size_t)b * N + k) * (size_t)ldc + j];
    }
    const float tf = ((1.0f - cosv) - nm.f_lo) * nm.f_rinv;
    const float dx = sqrtf(sqdist_rn(xj, yj, zj, X[3 * k], X[3 * k + 1], X[3 * k + 2]));
    const float tx = (dx - nm.x_lo) * nm.x_rinv;
    const int dt = tj - TAU[k];
    const float tt = dt > 0 ? (float)dt * nm.t_rinv : 0.0f;
    acc += P.alpha_f * tf + P.alpha_x * tx + P.alpha_tau * tt;
  }
  r_all[(size_t)b * N + j] = P.n_cap > 0 ? acc / (float)P.n_cap : 0.0f;
}

// v_j = r_j / sum_l r_l (phi = identity), uniform when the sum is 0 or the
// uniform-capacity ablation is on.  The sum is taken in fp64 in a fixed order
// (thread r adds j = r, r + 1024, ...).  Bound by the few fp64 units of an SM,
// a division taking ~15 of their operations: every block adds up the whole
// scene and divides `chunk` tokens of it.  One scene of 8192 / 16384 tokens
// 10 / 15 us; one block dividing all of them took 34 / 64.  32 scenes of 8192
// 26 (34).
__global__ void __launch_bounds__(1024) k_capacity_v(const float* __restrict__ r_all, int N,
                                                     int mode, int chunk,
                                                     float* __restrict__ v_all,
                                                     float* __restrict__ v_out) {
  const int b = blockIdx.y;
  const float* r = r_all + (size_t)b * N;
  double part = 0.0;
  for (int j0 = threadIdx.x; j0 < N; j0 += 4 * 1024) {
    float x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = j0 + 1024 * u < N ? r[j0 + 1024 * u] : 0.0f;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (j0 + 1024 * u < N) part += (double)x[u];
  }
  part = warp_sum(part);
  __shared__ double s_part[32];
  __shared__ double s_total;
  if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += s_part[i];
    s_total = t;
  }
  __syncthreads();
  const double total = s_total;
  const bool uniform = mode == 1 || !(total > 0.0);
  const int end = min(N, (int)(blockIdx.x + 1) * chunk);
  for (int j = blockIdx.x * chunk + threadIdx.x; j < end; j += blockDim.x) {
    const float vj = uniform ? (float)(1.0 / (double)N) : (float)((double)r[j] / total);
    v_all[(size_t)b * N + j] = vj;
    if (v_out) v_out[(size_t)b * N + j] = vj;
  }
}

int launch_capacity(const void* feats, int dtype, const float* inv, const float* pos,
                    const int32_t* frame, const SceneNorms* norms, const int32_t* nbr,
                    const DevParams& P, int64_t B, int64_t N, int64_t D, float* r, float* v,
                    float* v_out, cudaStream_t s, const float* cos, int64_t ldc,
                    const int32_t* pos_of, const float4* order) {
  // one block per token, a warp per neighbour (at most CAP_WARPS)
  const dim3 grid((unsigned)N, (unsigned)B);
  const int warps = P.n_cap < 1 ? 1 : (P.n_cap < CAP_WARPS ? P.n_cap : CAP_WARPS);
  // rows at a time: the last turn multiplies its row count whatever is left.
  // Lite of 8 scenes of 8192, D = 3584, us, 2 / 4 / 8 rows: 1 neighbour 573 / 613 /
  // 659 (a block a token 731), 2 576 / 619 / 662 (756), 3 625 / 623 / 674, 4 633 /
  // 628 / 681, 5 683 / 705 / 692, 6 689 / 711 / 703, 8 746 / 720 / 720, 9 798 / 799
  // / 852, 12 863 / 818 / 874, 13 915 / 895 / 885, 16 980 / 916 / 916.
  const auto near = P.n_cap <= 2                                     ? k_capacity_r_near<2>
                    : P.n_cap <= 4 || (P.n_cap > 8 && P.n_cap <= 12) ? k_capacity_r_near<4>
                                                                     : k_capacity_r_near<8>;
  if (cos)
    k_capacity_r_cos<<<dim3((unsigned)((N + 255) / 256), (unsigned)B), 256, 0, s>>>(
        cos, ldc, pos, frame, norms, nbr, P, (int)N, pos_of, r);
  else if (dtype == CP_BF16 && order)
    near<<<dim3((unsigned)((N + 7) / 8), (unsigned)B), 256, 0, s>>>(
        (const __nv_bfloat16*)feats, inv, pos, frame, norms, nbr, order, P, (int)N, (int)D, r);
  else if (dtype == CP_BF16)
    k_capacity_r<__nv_bfloat16><<<grid, 32 * warps, 0, s>>>(
        (const __nv_bfloat16*)feats, inv, pos, frame, norms, nbr, P, (int)N, (int)D, r);
  else
    k_capacity_r<float><<<grid, 32 * warps, 0, s>>>((const float*)feats, inv, pos, frame, norms,
                                                        nbr, P, (int)N, (int)D, r);
  int st = last_launch_status();
  if (st != CP_OK) return st;
  // chunks of 128 tokens while few scenes leave SMs idle, up to 1024
  DeviceInfo di;
  if (device_info(&di) != CP_OK) return CP_ECUDA;
  int chunk = 128;
  while (chunk < 1024 && B * ((N + chunk - 1) / chunk) > 2 * di.sm_count) chunk <<= 1;
  k_capacity_v<<<dim3((unsigned)((N + chunk - 1) / chunk), (unsigned)B), 1024, 0, s>>>(
      r, (int)N, P.cap_mode, chunk, v, v_out);
  return last_launch_status();
}

// slab[b][t][k] = C(t, M_g(t)[k]) with M_g(t)[0] = t and M_g(t)[k] the k-th
// nearest other token for k >= 1.
__global__ void k_slab(const float* __restrict__ cost, int64_t ldc, const int32_t* __restrict__ nbr,
                       int kk, int g, int N, float* __restrict__ slab) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int b = blockIdx.y;
  if (i >= (int64_t)N * g) return;
  const int t = (int)(i / g), k = (int)(i % g);
  const int j = k == 0 ? t : nbr[((size_t)b * N + t) * kk + (k - 1)];
  slab[(size_t)b * N * g + i] = cost[(size_t)b * N * ldc + (size_t)t * ldc + j];
}

int launch_slab(const float* cost, int64_t ldc, const int32_t* nbr, const DevParams& P, int64_t B,
                int64_t N, float* slab, cudaStream_t s) {
  const int64_t n = N * P.g;
  dim3 grid((unsigned)((n + 255) / 256), (unsigned)B);
  k_slab<<<grid, 256, 0, s>>>(cost, ldc, nbr, P.kk, P.g, (int)N, slab);
  return last_launch_status();
}

}  // namespace cp
