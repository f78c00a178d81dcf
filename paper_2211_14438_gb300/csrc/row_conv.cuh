// Row convolutions of the squaring step (a4, order 2): one output row of the
// square of a polynomial held in row layout (monomials sharing the exponents
// of t_1..t_{n-1} contiguous), as the sum of 1-D convolutions of input-row
// pairs, unrolled for every pair of row lengths up to kRowLen, for the fused
// layer kernel (k_layer.cu).
#pragma once

#include "device_util.cuh"

namespace bern {

// One accumulator per output slot holds the square directly: an off-diagonal
// row pair (p < q) counts twice in the square, so it multiplies 2*x[a]
// (exact) by y[b]; the diagonal pair (p == q) is the row's own square,
// sum_a x[a]^2 t^(2a) + sum_(a<b) 2 x[a] x[b] t^(a+b), taken as a triangle.
// A per-lane sign sg = +1 or -1 multiplies the first operand, and every FMA
// rounds up.  With sg = -1 every partial sum is the exact negation
// of the round-down one (RU(-x) = -RD(x) in IEEE arithmetic), so lanes that
// compute the lower bound (sg = -1) and lanes that compute the upper bound
// (sg = +1) run the same instructions.
template <int L1, int L2>
__device__ __forceinline__ void conv_rows_sg(const float* __restrict__ s, int offp, int offq,
                                             float sg2, float (&acc)[2 * kRowLen - 1]) {
  float x[L1], y[L2];
#pragma unroll
  for (int a = 0; a < L1; ++a) x[a] = s[offp + a] * sg2;   // +-2 s: exact
#pragma unroll
  for (int b = 0; b < L2; ++b) y[b] = s[offq + b];
#pragma unroll
  for (int a = 0; a < L1; ++a)
#pragma unroll
    for (int b = 0; b < L2; ++b) acc[a + b] = __fmaf_ru(x[a], y[b], acc[a + b]);
}

template <int L>
__device__ __forceinline__ void conv_diag_sg(const float* __restrict__ s, int off, float sg,
                                             float (&acc)[2 * kRowLen - 1]) {
  float x[L], xs[L], x2[L];
#pragma unroll
  for (int a = 0; a < L; ++a) {
    x[a] = s[off + a];
    xs[a] = x[a] * sg;
    x2[a] = xs[a] + xs[a];
  }
#pragma unroll
  for (int a = 0; a < L; ++a) {
    acc[2 * a] = __fmaf_ru(xs[a], x[a], acc[2 * a]);
#pragma unroll
    for (int b = a + 1; b < L; ++b) acc[a + b] = __fmaf_ru(x2[a], x[b], acc[a + b]);
  }
}

#define BERN_CCS(L1, L2) \
  case row_pair_case(L1, L2): conv_rows_sg<L1, L2>(s, pr.x, pr.y, sg2, acc); break;
#define BERN_CONV_SG_CASES                                                                     \
  BERN_CCS(1, 1) BERN_CCS(1, 2) BERN_CCS(1, 3) BERN_CCS(1, 4) BERN_CCS(1, 5) BERN_CCS(1, 6)    \
  BERN_CCS(1, 7) BERN_CCS(1, 8) BERN_CCS(1, 9) BERN_CCS(2, 2) BERN_CCS(2, 3) BERN_CCS(2, 4)    \
  BERN_CCS(2, 5) BERN_CCS(2, 6) BERN_CCS(2, 7) BERN_CCS(2, 8) BERN_CCS(2, 9) BERN_CCS(3, 3)    \
  BERN_CCS(3, 4) BERN_CCS(3, 5) BERN_CCS(3, 6) BERN_CCS(3, 7) BERN_CCS(3, 8) BERN_CCS(3, 9)    \
  BERN_CCS(4, 4) BERN_CCS(4, 5) BERN_CCS(4, 6) BERN_CCS(4, 7) BERN_CCS(4, 8) BERN_CCS(4, 9)    \
  BERN_CCS(5, 5) BERN_CCS(5, 6) BERN_CCS(5, 7) BERN_CCS(5, 8) BERN_CCS(5, 9) BERN_CCS(6, 6)    \
  BERN_CCS(6, 7) BERN_CCS(6, 8) BERN_CCS(6, 9) BERN_CCS(7, 7) BERN_CCS(7, 8) BERN_CCS(7, 9)    \
  BERN_CCS(8, 8) BERN_CCS(8, 9) BERN_CCS(9, 9)
#define BERN_CDS(L) \
  case L: conv_diag_sg<L>(s, pr.x, sg, acc); break;
#define BERN_DIAG_SG_CASES \
  BERN_CDS(1) BERN_CDS(2) BERN_CDS(3) BERN_CDS(4) BERN_CDS(5) BERN_CDS(6) BERN_CDS(7) BERN_CDS(8) \
  BERN_CDS(9)

}  // namespace bern
