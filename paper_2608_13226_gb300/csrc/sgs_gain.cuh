// The gain of the greedy selection (Sec. 3.5) as every selection kernel
// computes it:
//     gain(t) = sum_{j in M_g(t)} v_j max(m_j - C(t, j), 0).
//
// A term is v_j * max(m_j - C, 0) in fp32, each operation rounded once, and
// the terms add up in 64-bit fixed point: term -> floor(term 2^S), with 2^S
// chosen so that the largest possible gain stays below 2^62.  Integer
// addition has no rounding and no order, so a gain is the same number however
// it is computed: summed over a row, over a list, over several blocks, or
// kept up to date by subtracting what a pick took away from single terms.
// Every term is non-increasing in m, so gains are non-increasing too.
//
// The scale follows the gains, not m0, which may be any number: it starts
// from m0 (sum v = 1), on the dense path from the largest cost once the first
// pick has covered every target (gain_fx_covered), and whenever the best
// gain left is below 2^-24 of it, it is fitted to that gain and the gains are
// summed afresh before the pick (gain_floor, gain_refit; at most 8 times in a
// selection, as it falls by 2^24 or more each time).  A term loses at most
// 2^-60 of the scale, so n terms 2^-36 n of the best gain.
//
// Decisions and recorded gains use the sum rounded to 24 bits, an fp32 number
// (equal sums give equal numbers and larger sums never smaller ones); the
// lowest index wins among equal ones.  Against 64-bit sums of the same costs
// the recorded gains of a selection of 8192 tokens are off by 2.8e-8 of their
// norm and none by more than 8.6e-8; fp32 sums of the same terms, kept
// before, by 3.9e-8 and 1.2e-7.
#pragma once

#include "common.cuh"

namespace cp {

typedef unsigned long long gain_t;  // a gain or a term, in units of 2^-S

// floor(p 2^S) of a term p >= 0, with S = 190 - fx (fx from gain_fx below).
// The mantissa with its leading one sits at the top of a 64-bit word and is
// shifted down by fx - exponent; shr.u64 takes shifts past 63 as 64, so zero
// (exponent field 0, and fx >= 64) gives 0.
__device__ __forceinline__ gain_t fixed_term(float p, int fx) {
  const uint32_t b = __float_as_uint(p);
  const uint32_t top = (b << 8) | 0x80000000u;
  gain_t r;
  asm("{\n\t.reg .b64 x;\n\tmov.b64 x, {%3, %1};\n\tshr.u64 %0, x, %2;\n\t}"
      : "=l"(r)
      : "r"(top), "r"((uint32_t)fx - (b >> 23)), "r"(0u));
  return r;
}
__device__ __forceinline__ gain_t gain_term(float v, float m, float c, int fx) {
  return fixed_term(__fmul_rn(v, fmaxf(__fsub_rn(m, c), 0.0f)), fx);
}

// What lowering m_j from mo to mn takes off the term.
__device__ __forceinline__ gain_t gain_drop(float v, float mo, float mn, float c, int fx) {
  return gain_term(v, mo, c, fx) - gain_term(v, mn, c, fx);
}

// A gain rounded to 24 bits, as fp32 bits (0 for 0; fx >= 64).
__device__ __forceinline__ uint32_t gain_bits(gain_t g, int fx) {
  if (g == 0ull) return 0u;
  const int lz = __clzll((long long)g);
  return ((uint32_t)(fx - lz - 1) << 23) + (((uint32_t)((g << lz) >> 39) + 1u) >> 1);
}

// The refit of the scale, a rule on the best gain left that every selection
// kernel applies at the same step.  gain_floor: its 24 bits below which the
// scale no longer fits; gain_refit: the scale that does.  Before their cut
// the sums of up to 2^lgN terms are below that gain and 2^lgN units together.
__device__ __forceinline__ uint32_t gain_floor(int fx) {
  return fx > 64 ? (uint32_t)(fx - 27) << 23 : 0u;
}
__device__ __forceinline__ int gain_refit(uint32_t bits, int fx, int lgN) {
  const int of_gain = bits ? (int)(bits >> 23) + 4 : 64, of_cut = fx - 60 + lgN;
  return max(64, max(of_gain, of_cut));
}

// (gain, index) as one key: the largest gain wins, the lowest index among
// equal gains; 0 is below every candidate.
__device__ __forceinline__ gain_t gain_key(uint32_t bits, int t) {
  return ((gain_t)(bits + 1u) << 32) | (0xFFFFFFFFu - (uint32_t)t);
}
__device__ __forceinline__ int key_token(gain_t key) {
  return (int)(0xFFFFFFFFu - (uint32_t)(key & 0xFFFFFFFFull));
}
__device__ __forceinline__ float key_gain(gain_t key) {
  return __uint_as_float((uint32_t)(key >> 32) - 1u);
}

// The warp's sum of 62-bit values, as three 32-bit reductions of 27-bit parts
// (32 of them stay below 2^32): half the instructions of a 64-bit butterfly.
__device__ __forceinline__ gain_t warp_sum_gain(gain_t v) {
  const uint32_t a = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)v & 0x7FFFFFFu);
  const uint32_t b = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)(v >> 27) & 0x7FFFFFFu);
  const uint32_t c = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)(v >> 54));
  return (gain_t)a + ((gain_t)b << 27) + ((gain_t)c << 54);
}
// The largest key of the warp, by two 32-bit reductions.
__device__ __forceinline__ gain_t warp_max_key(gain_t k) {
  const uint32_t hi = (uint32_t)(k >> 32);
  const uint32_t mh = __reduce_max_sync(0xFFFFFFFFu, hi);
  const uint32_t ml = __reduce_max_sync(0xFFFFFFFFu, hi == mh ? (uint32_t)k : 0u);
  return ((gain_t)mh << 32) | ml;
}

__device__ __forceinline__ float4 ld_stream_f4(const float4* p) {
  float4 r;
  asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w)
               : "l"(p));
  return r;
}

// gain(t) over a dense padded row by one warp (pad columns: v = 0): 16-byte
// loads, eight in flight a lane.  A group of 128 columns without any C < m
// holds only zero terms and skips the arithmetic (the sweep is bound by HBM
// only if most groups do: the fixed-point sum takes ~12 instructions a
// column, against 3 of the fp32 sum it replaced).
__device__ __forceinline__ gain_t dense_row_gain(const float* __restrict__ crow, const float* m,
                                                 const float* v, int ncols, int fx, int lane) {
  const float4* row = reinterpret_cast<const float4*>(crow);
  const float4* m4 = reinterpret_cast<const float4*>(m);
  const float4* v4 = reinterpret_cast<const float4*>(v);
  const int nq = ncols >> 2;
  gain_t acc = 0ull;
  for (int i0 = lane; i0 - lane < nq; i0 += 8 * 32) {
    float4 cs[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      cs[u] = i0 + 32 * u < nq ? ld_stream_f4(row + i0 + 32 * u)
                               : make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = i0 + 32 * u;
      const float4 c = cs[u];
      const float4 mm = i < nq ? m4[i] : make_float4(0.f, 0.f, 0.f, 0.f);
      const bool live = c.x < mm.x || c.y < mm.y || c.z < mm.z || c.w < mm.w;
      if (!__any_sync(0xFFFFFFFFu, live)) continue;
      const float4 vv = i < nq ? v4[i] : make_float4(0.f, 0.f, 0.f, 0.f);
      acc += gain_term(vv.x, mm.x, c.x, fx);
      acc += gain_term(vv.y, mm.y, c.y, fx);
      acc += gain_term(vv.z, mm.z, c.z, fx);
      acc += gain_term(vv.w, mm.w, c.w, fx);
    }
  }
  return warp_sum_gain(acc);
}

// gain(t) over the local neighbourhood M_g(t) by one warp: a slab row of g
// costs, member 0 is t itself, members k >= 1 are t's nearest others.  Bound
// by instruction issue: the first 64 members go without a bounds check (300
// steps of 8 scenes of 8192, g = 64: 5.1 ms, 5.4 with one).
__device__ __forceinline__ gain_t local_row_gain(const float* __restrict__ srow,
                                                 const int32_t* __restrict__ nb, int t, int g,
                                                 const float* sm_m, const float* sm_v, int fx,
                                                 int lane) {
  gain_t acc = 0ull;
  int k = lane;
  if (g >= 64) {
    const int j0 = k > 0 ? nb[k - 1] : t, j1 = nb[k + 31];
    const float c0 = srow[k], c1 = srow[k + 32];
    acc = gain_term(sm_v[j0], sm_m[j0], c0, fx) + gain_term(sm_v[j1], sm_m[j1], c1, fx);
    k += 64;
  }
#pragma unroll 1
  for (; k < g; k += 32) {
    const int j = k > 0 ? nb[k - 1] : t;
    acc += gain_term(sm_v[j], sm_m[j], srow[k], fx);
  }
  return warp_sum_gain(acc);
}

// F(S) = sum_j v_j m_j in fp64, in one fixed order whatever the block size
// (>= 512 threads): thread r < 512 sums j = r, r+512, ...; then 16 warp
// butterflies; then the 16 warp sums in order.  Every thread of the block
// must call it; the result is valid in thread 0.
__device__ __forceinline__ double objective_sum(const float* m, const float* v, int N) {
  __shared__ double s_part[16];
  double part = 0.0;
  if (threadIdx.x < 512)
    for (int j = threadIdx.x; j < N; j += 512) part += (double)v[j] * (double)m[j];
  if (threadIdx.x < 512) part = warp_sum(part);
  if (threadIdx.x < 512 && (threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = part;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < 16; ++i) t += s_part[i];
  return t;
}

}  // namespace cp
