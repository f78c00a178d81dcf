// Device helpers: directed rounding, block reductions, binomial tables.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "bern_internal.cuh"

namespace bern {

// UP = round towards +inf (upper bounds), !UP = towards -inf (lower bounds)
template <bool UP>
__device__ __forceinline__ float dfma(float a, float b, float c) {
  return UP ? __fmaf_ru(a, b, c) : __fmaf_rd(a, b, c);
}
template <bool UP>
__device__ __forceinline__ float dadd(float a, float b) {
  return UP ? __fadd_ru(a, b) : __fadd_rd(a, b);
}

// warp-wide directed sum (fixed tree: deterministic)
template <bool UP>
__device__ __forceinline__ float warp_dsum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = dadd<UP>(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float warp_min(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ int warp_imax(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Block-wide directed sum; scratch holds >= 32 floats; all threads get the
// result.  Must be called by every thread of the block.
template <bool UP>
__device__ float block_dsum(float v, float* scratch) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nw = (blockDim.x + 31) >> 5;
  v = warp_dsum<UP>(v);
  __syncthreads();
  if (lane == 0) scratch[wid] = v;
  __syncthreads();
  float r = lane < nw ? scratch[lane] : 0.0f;
  r = warp_dsum<UP>(r);
  return r;
}

// Appends the block's items to NQ work lists in item order (q: the thread's list,
// -1 none): the rank of equal lists within a warp, a scan over the warps by one
// warp per list, one atomic per list and block.  Called by every thread of a block
// of whole warps.
template <int NQ>
__device__ __forceinline__ void append_to_lists(int q, int item, int* qcount, int32_t* queue,
                                                int64_t qcap) {
  constexpr int S = NQ | 1;                  // odd stride: a list's column without conflicts
  __shared__ int s_at[32 * S];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int i = threadIdx.x; i < 32 * S; i += blockDim.x) s_at[i] = 0;
  __syncthreads();
  const unsigned same = __match_any_sync(0xffffffffu, q);
  const int rank = __popc(same & ((1u << lane) - 1u));
  if (q >= 0 && rank == 0) s_at[warp * S + q] = __popc(same);
  __syncthreads();
  for (int l = warp; l < NQ; l += nw) {
    const int c = s_at[lane * S + l];
    int run = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, run, o);
      if (lane >= o) run += v;
    }
    int base = 0;
    if (lane == 31 && run) base = atomicAdd(&qcount[l], run);
    s_at[lane * S + l] = __shfl_sync(0xffffffffu, base, 31) + run - c;
  }
  __syncthreads();
  if (q >= 0) queue[(int64_t)q * qcap + s_at[warp * S + q] + rank] = item;
}

// Exact binomials C(l,k), l,k <= 24 (all < 2^24, so exact in float32).
struct BinomTable {
  float v[kMaxEncloseOrder + 1][kMaxEncloseOrder + 1];
};
constexpr BinomTable make_binom_table() {
  BinomTable t{};
  for (int l = 0; l <= kMaxEncloseOrder; ++l) {
    t.v[l][0] = 1.0f;
    for (int k = 1; k <= l; ++k) t.v[l][k] = t.v[l - 1][k - 1] + (k <= l - 1 ? t.v[l - 1][k] : 0.0f);
  }
  return t;
}
__constant__ const BinomTable c_binom = make_binom_table();

__device__ __forceinline__ float binomf(int l, int k) { return c_binom.v[l][k]; }


}  // namespace bern
