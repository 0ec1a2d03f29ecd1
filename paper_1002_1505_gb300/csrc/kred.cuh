// Per-RHS reductions for kernels whose CTAs are laid out by the FFT passes
// rather than by a vector loop: each CTA reduces its products into one slot of
// a partial-sum table, and the last CTA of a right-hand side to arrive (a
// device-scope counter) sums that RHS's slots in a fixed order.  The scheme and
// the double-float product accumulation of a thread are those of the Krylov
// vector kernels (krylov.cu); across a warp those add in FP64 and the folded
// passes in three floats (sum3.cuh), so the two differ in the last bits of FP64.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "dda_internal.h"
#include "sum3.cuh"

namespace dda {
namespace kred {

// Two running sums of float products side by side, each carried as a double-float pair (products split
// exactly with one FMA, added with the two-sum), on the packed FP32 instructions: conj(a) b as (re, im),
// or the two squares of |a|^2.
struct AccF2 {
  float2 hi = {0.f, 0.f}, lo = {0.f, 0.f};
  __device__ __forceinline__ void fma(float2 a, float2 b) {
    auto neg = [](float2 v) { return make_float2(-v.x, -v.y); };
    const float2 p = __fmul2_rn(a, b);
    const float2 pe = __ffma2_rn(a, b, neg(p));
    const float2 t = __fadd2_rn(hi, p);
    const float2 z = __fadd2_rn(t, neg(hi));
    const float2 e = __fadd2_rn(__fadd2_rn(hi, neg(__fadd2_rn(t, neg(z)))), __fadd2_rn(p, neg(z)));
    hi = t;
    lo = __fadd2_rn(lo, __fadd2_rn(e, pe));
  }
};
__device__ __forceinline__ void acc_cdot(AccF2& c, float2 a, float2 b) {
  c.fma(make_float2(a.x, a.x), b);
  c.fma(make_float2(a.y, a.y), make_float2(b.y, -b.x));
}
__device__ __forceinline__ void acc_nrm(AccF2& s, float2 a) { s.fma(a, a); }

// (h, l) += (h2, l2), sums carried as double-float pairs
__device__ __forceinline__ void pair_add(float& h, float& l, float h2, float l2) {
  const float s = __fadd_rn(h, h2), z = __fsub_rn(s, h);
  l = __fadd_rn(__fadd_rn(l, l2), __fadd_rn(__fsub_rn(h, __fsub_rn(s, z)), __fsub_rn(h2, z)));
  h = s;
}

// Block sum of NS pairs, blockDim.x = 256.  The warps' sums are carried in three floats (Sum3), which keep
// more than the FP64 shuffle tree that they stand for: that tree runs at 1/64 of the FP32 rate and costs a
// CTA 1900 issue cycles for three values of eight warps.  (A tree of pairs keeps fewer bits than FP64, and
// three floats cost next to nothing more: a 64 x 48 x 32 solve takes 4.169 ms with them, 4.163 with pairs.)
// Then one warp turns the eight warps' sums of all values into FP64 and adds them; result in out (doubles,
// NS <= 4).  Lanes 0, 8, .. of that warp store a value each; its closing __syncwarp orders their stores
// before whatever thread 0 does next, so that a fence and a release by thread 0 alone publish all of them.
template <int NS>
__device__ __forceinline__ void block_sum_pairs(float (&h)[NS], float (&l)[NS], double* out) {
  __shared__ Sum3 red[NS * 8];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    Sum3 v{h[s], l[s], 0.f};
    for (int o = 16; o > 0; o >>= 1)
      v.add(Sum3{__shfl_down_sync(0xffffffffu, v.h, o), __shfl_down_sync(0xffffffffu, v.l, o),
                 __shfl_down_sync(0xffffffffu, v.t, o)});
    if (lane == 0) red[s * 8 + w] = v;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    double x = threadIdx.x < NS * 8 ? red[threadIdx.x].get() : 0.0;
    for (int o = 4; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o, 8);
    if (threadIdx.x % 8 == 0 && threadIdx.x < NS * 8) out[threadIdx.x / 8] = x;
    __syncwarp();
  }
}

// Block sum of v (all threads call; blockDim.x a multiple of 32, at most 1024); result in out (thread 0 writes).
template <int NS>
__device__ __forceinline__ void block_sum(double (&v)[NS], double* out) {
  __shared__ double red[NS][32];
#pragma unroll
  for (int s = 0; s < NS; ++s)
    for (int o = 16; o > 0; o >>= 1) v[s] += __shfl_down_sync(0xffffffffu, v[s], o);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0)
#pragma unroll
    for (int s = 0; s < NS; ++s) red[s][w] = v[s];
  __syncthreads();
  if (threadIdx.x < 32) {
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      double x = (threadIdx.x < (blockDim.x >> 5)) ? red[s][threadIdx.x] : 0.0;
      for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
      if (threadIdx.x == 0) out[s] = x;
    }
  }
}

// Store this CTA's block sum of the pairs (h, l) in slot `slot` of RHS b (nblk slots per RHS, kRedSlots
// doubles each).  Returns true in every thread of the last CTA of b to arrive, with b's totals
// in tot; that CTA also resets b's counter to zero.  All threads of the CTA must call it.
template <int NS>
__device__ __forceinline__ bool last_cta_totals(float (&h)[NS], float (&l)[NS], double* part, unsigned int* count,
                                                int b, int slot, int nblk, double (&tot)[NS]) {
  double* mine = part + ((int64_t)b * nblk + slot) * kRedSlots;
  block_sum_pairs<NS>(h, l, mine);
  __shared__ unsigned int s_last;
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = (atomicAdd(count + b, 1u) == (unsigned)nblk - 1u) ? 1u : 0u;
  }
  __syncthreads();
  if (!s_last) return false;
  __threadfence();
  const double* base = part + (int64_t)b * nblk * kRedSlots;
  double v[NS];
#pragma unroll
  for (int q = 0; q < NS; ++q) v[q] = 0.0;
  for (int i = threadIdx.x; i < nblk; i += blockDim.x)
#pragma unroll
    for (int q = 0; q < NS; ++q) v[q] += __ldcg(base + (int64_t)i * kRedSlots + q);
  __shared__ double res[NS];
  block_sum<NS>(v, res);
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NS; ++q) tot[q] = res[q];
  if (threadIdx.x == 0) count[b] = 0;
  return true;
}

__device__ __forceinline__ double2 cdiv(double2 a, double2 b) {
  const double d = b.x * b.x + b.y * b.y;
  return make_double2((a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d);
}

}  // namespace kred
}  // namespace dda
