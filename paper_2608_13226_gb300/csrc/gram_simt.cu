// K2/K3 for fp32 features (bf16 features use gram_tc.cu): Gram tiles with fp32
// FMA (TF32 tensor cores would round the features to 10 mantissa bits, far
// outside the fp32 tolerance) over the tiles touching i <= j: the max and min
// of cos(f_i, f_j) (the feature normaliser of Sec. 3.3) and, with an output
// buffer, the dot products themselves at [i][j].  Once the normalisers are
// known, one pass over them (k_fst_simt) writes the FST cost of Eq. fst_cost
// of (i, j) and of (j, i).
// A TM x TM output tile per 256-thread block, (TM / 16)^2 outputs a thread, K
// chunks of 16 staged through shared memory.  TM = 128 unless its tiles leave
// SMs without one: 1024 tokens, D = 256, 36 tiles of 128 or 136 of 64.
// Bound by the FMA rate where the tiles fill the device.  A second Gram over
// all tiles with the cost as its epilogue, the form before, made three times
// the products: 1024 tokens, D = 256 24 + 12 us, 48 + 76 before; the whole
// cost call of 3000 tokens, D = 512 0.24 ms (0.54), of 8 such scenes 1.46
// (3.18).
#include "common.cuh"

namespace cp {

constexpr int ST_BK = 16, ST_THREADS = 256;

template <int TM>
__device__ __forceinline__ void stage_tile(const float* __restrict__ F, int row0, int N, int D,
                                           int k0, float (*S)[TM + 4]) {
  constexpr int PER_ROW = ST_BK / 4;  // 16-byte loads per row per chunk
  for (int i = threadIdx.x; i < TM * PER_ROW; i += ST_THREADS) {
    const int r = i / PER_ROW, c = (i % PER_ROW) * 4;
    const int gr = row0 + r, gc = k0 + c;
    float x[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (gr < N && gc < D) Vec16<float>::load(F + (size_t)gr * D + gc, x);
#pragma unroll
    for (int q = 0; q < 4; ++q) S[c + q][r] = x[q];
  }
}

template <int TM>
__global__ void __launch_bounds__(ST_THREADS) k_gram_simt(
    const float* __restrict__ F_all, const float* __restrict__ inv_all, int N, int D,
    float* __restrict__ dots, int64_t ldc, SceneStats* stats) {
  constexpr int R = TM / 16;  // outputs a thread and axis, in groups of four
  const int b = blockIdx.z;
  const int row0 = blockIdx.y * TM, col0 = blockIdx.x * TM;
  if (col0 < row0) return;  // only pairs j < i inside
  const float* F = F_all + (size_t)b * N * D;
  const float* inv = inv_all + (size_t)b * N;

  __shared__ __align__(16) float As[ST_BK][TM + 4];
  __shared__ __align__(16) float Bs[ST_BK][TM + 4];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float acc[R][R];
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int j = 0; j < R; ++j) acc[i][j] = 0.0f;

  for (int k0 = 0; k0 < D; k0 += ST_BK) {
    stage_tile<TM>(F, row0, N, D, k0, As);
    stage_tile<TM>(F, col0, N, D, k0, Bs);
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < ST_BK; ++kk) {
      float a[R], bb[R];
#pragma unroll
      for (int h = 0; h < R; h += 4) {
        const float4 x = *reinterpret_cast<const float4*>(&As[kk][16 * h + ty * 4]);
        const float4 y = *reinterpret_cast<const float4*>(&Bs[kk][16 * h + tx * 4]);
        a[h] = x.x; a[h + 1] = x.y; a[h + 2] = x.z; a[h + 3] = x.w;
        bb[h] = y.x; bb[h + 1] = y.y; bb[h + 2] = y.z; bb[h + 3] = y.w;
      }
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j) acc[i][j] = fmaf(a[i], bb[j], acc[i][j]);
    }
    __syncthreads();
  }

  float cmax = -INFINITY, cmin = INFINITY;
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int gi = row0 + 16 * (i & ~3) + ty * 4 + (i & 3);
    if (gi >= N) continue;
    const float inv_i = inv[gi];
    float* row = dots ? dots + ((size_t)b * N + gi) * (size_t)ldc : nullptr;
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int gj = col0 + 16 * (j & ~3) + tx * 4 + (j & 3);
      if (gj >= N) continue;
      if (row) row[gj] = acc[i][j];
      float c = clamp_cos(acc[i][j] * inv_i * inv[gj]);
      if (gi == gj && inv_i > 0.0f) c = 1.0f;  // cos(f, f) = 1 exactly
      cmax = fmaxf(cmax, c);
      cmin = fminf(cmin, c);
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    cmax = fmaxf(cmax, __shfl_xor_sync(0xFFFFFFFFu, cmax, o));
    cmin = fminf(cmin, __shfl_xor_sync(0xFFFFFFFFu, cmin, o));
  }
  if ((threadIdx.x & 31) == 0 && cmax >= cmin) {
    atomicMax(&stats[b].cos_max_key, f2key(cmax));
    atomicMin(&stats[b].cos_min_key, f2key(cmin));
  }
}

// The cost from the stored dot products, in place: the block of tile (I, J),
// I <= J, reads it and writes tiles (I, J) and (J, I).  Pad columns get 0.
// 1024 threads a tile: 1024 tokens 12 us (256: 19), 8 scenes of 3000 4% more of
// the call than with 256.
constexpr int FS_T = 64, FS_THREADS = 1024, FS_STEP = FS_THREADS / FS_T;
__global__ void __launch_bounds__(FS_THREADS) k_fst_simt(float* __restrict__ cost, int64_t ldc, int N,
                                                  const float* __restrict__ inv_all,
                                                  const float* __restrict__ pos_all,
                                                  const int32_t* __restrict__ frame_all,
                                                  const SceneNorms* __restrict__ norms,
                                                  DevParams P) {
  const int J = blockIdx.x, I = blockIdx.y, b = blockIdx.z;
  if (J < I) return;
  __shared__ float s_dot[FS_T][FS_T + 1];
  __shared__ float s_inv[2][FS_T], s_x[2][3][FS_T];  // tile I's tokens, tile J's
  __shared__ int s_t[2][FS_T];
  float* C = cost + (size_t)b * N * (size_t)ldc;
  const SceneNorms nm = norms[b];
  if (threadIdx.x < 2 * FS_T) {
    const int h = threadIdx.x / FS_T, r = threadIdx.x % FS_T;
    const int t = min((h ? J : I) * FS_T + r, N - 1);
    s_inv[h][r] = inv_all[(size_t)b * N + t];
#pragma unroll
    for (int a = 0; a < 3; ++a) s_x[h][a][r] = pos_all[((size_t)b * N + t) * 3 + a];
    s_t[h][r] = frame_all[(size_t)b * N + t];
  }
  const int c = threadIdx.x % FS_T, r0 = threadIdx.x / FS_T;
  for (int r = r0; r < FS_T; r += FS_STEP)
    if (I * FS_T + r < N && J * FS_T + c < N)
      s_dot[r][c] = C[(size_t)(I * FS_T + r) * ldc + J * FS_T + c];
  __syncthreads();
  // token r of side h against token c of the other side
  auto one = [&](int h, int r, int c, float dot, bool same) -> float {
    const int o = h ^ 1;
    float cosv = clamp_cos(dot * s_inv[h][r] * s_inv[o][c]);
    if (same && s_inv[h][r] > 0.0f) cosv = 1.0f;  // cos(f, f) = 1 exactly
    const float d2 = sqdist_rn(s_x[h][0][r], s_x[h][1][r], s_x[h][2][r], s_x[o][0][c],
                               s_x[o][1][c], s_x[o][2][c]);
    return fst_cost_from(cosv, d2, s_t[h][r], s_t[o][c], nm, P);
  };
  for (int r = r0; r < FS_T; r += FS_STEP) {
    const int i = I * FS_T + r, j = J * FS_T + c;
    if (i >= N || j >= ldc) continue;
    const float dot = I == J && c < r ? s_dot[c][r] : s_dot[r][c];
    C[(size_t)i * ldc + j] = j < N ? one(0, r, c, dot, i == j) : 0.0f;
  }
  if (I < J)
    for (int r = r0; r < FS_T; r += FS_STEP)
      if (J * FS_T + r < N)
        C[(size_t)(J * FS_T + r) * ldc + I * FS_T + c] = one(1, r, c, s_dot[c][r], false);
}

// dots (may be null): every dot product of a pair i <= j, [B][N][ldc].
int launch_gram_minmax_simt(const void* feats, int dtype, const float* inv, int64_t B, int64_t N,
                            int64_t D, SceneStats* stats, cudaStream_t s, float* dots,
                            int64_t ldc) {
  if (dtype != CP_F32) return CP_EINVAL;  // bf16 features run on the tensor cores
  DeviceInfo di;
  if (device_info(&di) != CP_OK) return CP_ECUDA;
  const int64_t n128 = (N + 127) / 128, n64 = (N + 63) / 64;
  if (B * n128 * (n128 + 1) / 2 < di.sm_count)
    k_gram_simt<64><<<dim3((unsigned)n64, (unsigned)n64, (unsigned)B), ST_THREADS, 0, s>>>(
        (const float*)feats, inv, (int)N, (int)D, dots, ldc, stats);
  else
    k_gram_simt<128><<<dim3((unsigned)n128, (unsigned)n128, (unsigned)B), ST_THREADS, 0, s>>>(
        (const float*)feats, inv, (int)N, (int)D, dots, ldc, stats);
  return last_launch_status();
}

int launch_fst_simt(float* cost, int64_t ldc, int64_t B, int64_t N, const float* inv,
                    const float* pos, const int32_t* frame, const SceneNorms* norms,
                    const DevParams& P, cudaStream_t s) {
  const unsigned T = (unsigned)((ldc + FS_T - 1) / FS_T);
  k_fst_simt<<<dim3(T, T, (unsigned)B), FS_THREADS, 0, s>>>(cost, ldc, (int)N, inv, pos, frame, norms, P);
  return last_launch_status();
}

}  // namespace cp
