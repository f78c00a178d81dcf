// The last two passes of the Bernstein enclosure in a thread's registers,
// shared by the two- and three-variable kernels (k_enclose_tail.cu) and the
// slab kernel of four and more variables (k_enclose_slab.cu).  Values are
// pairs (negated lower, upper polynomial), packed.cuh.
#pragma once

#include "enclose_impl.cuh"
#include "packed.cuh"

namespace bern {

// Largest order of the register passes of two and three variables: 45 pairs
// of coefficients at order 8 (66 at order 10, the slab kernel's largest).
constexpr int kTailMaxOrder = 8;

// Lexicographic order of the exponents of total degree <= l, the last exponent
// running: the offset of row j_1 among those of (j_1, j_2), and of row
// (j_1, j_2) among those of (j_1, j_2, j_3).
__host__ __device__ constexpr int lex2(int l, int j1) { return j1 * (l + 1) - j1 * (j1 - 1) / 2; }
__host__ __device__ constexpr int lex3(int l, int j1, int j2) {
  return ((l + 1) * (l + 2) * (l + 3) - (l - j1 + 1) * (l - j1 + 2) * (l - j1 + 3)) / 6 +
         lex2(l - j1, j2);
}

// A float as an int of the same order (for atomicMax), and back.
__device__ __forceinline__ int float_key(float x) {
  const int i = __float_as_int(x);
  return i >= 0 ? i : i ^ 0x7fffffff;
}
__device__ __forceinline__ float key_float(int k) {
  return __int_as_float(k >= 0 ? k : k ^ 0x7fffffff);
}

// line_transform_inplace on pairs: the same FMAs in the same order (a weight
// of one is an add: fma(1, x, y) = x + y).
template <int LB>
__device__ __forceinline__ void pair_transform(p2 (&x)[LB + 1]) {
#pragma unroll
  for (int i = LB; i >= 1; --i) {
    p2 acc = x[0];
#pragma unroll
    for (int j = 1; j <= i; ++j)
      acc = i == j ? add2_ru(x[j], acc) : fma2_ru(pack2(cbin(i, j), cbin(i, j)), x[j], acc);
    x[i] = acc;
  }
}

// The largest coefficients of a pair of polynomials in t_1, t_2 (scaled
// coefficients q in lexicographic order): the pass of t_2 one digit at a time,
// each followed by the pass of t_1 over its l + 1 values.
template <int LB>
__device__ __forceinline__ void pair_max(const p2 (&q)[(LB + 1) * (LB + 2) / 2], float& best_l,
                                         float& best_u) {
#pragma unroll
  for (int i2 = 0; i2 <= LB; ++i2) {
    p2 x[LB + 1];
#pragma unroll
    for (int j1 = 0; j1 <= LB; ++j1) {
      p2 acc = q[lex2(LB, j1)];
#pragma unroll
      for (int j2 = 1; j2 <= (i2 < LB - j1 ? i2 : LB - j1); ++j2)
        acc = i2 == j2 ? add2_ru(q[lex2(LB, j1) + j2], acc)
                       : fma2_ru(pack2(cbin(i2, j2), cbin(i2, j2)), q[lex2(LB, j1) + j2], acc);
      x[j1] = acc;
    }
    pair_transform<LB>(x);
#pragma unroll
    for (int i = 0; i <= LB; ++i) {
      float l, u;
      unpack2(x[i], l, u);
      best_l = fmaxf(best_l, l);
      best_u = fmaxf(best_u, u);
    }
  }
}

// The same of polynomials in t_1, t_2, t_3 at digit i3 of t_3: C their scaled
// coefficients in lexicographic order, bin the binomials [l+1][l+1] in shared
// memory (the digit differs between the lanes).
template <int LB>
__device__ __forceinline__ void tail_max(const p2* __restrict__ C, int i3,
                                         const p2* __restrict__ bin, float& best_l,
                                         float& best_u) {
  p2 q[(LB + 1) * (LB + 2) / 2];
#pragma unroll
  for (int j1 = 0; j1 <= LB; ++j1)
#pragma unroll
    for (int j2 = 0; j2 <= LB - j1; ++j2) q[lex2(LB, j1) + j2] = C[lex3(LB, j1, j2)];
#pragma unroll
  for (int j3 = 1; j3 <= LB; ++j3) {
    if (j3 <= i3) {
      const p2 w = bin[i3 * (LB + 1) + j3];
#pragma unroll
      for (int j1 = 0; j1 <= LB - j3; ++j1)
#pragma unroll
        for (int j2 = 0; j2 <= LB - j3 - j1; ++j2)
          q[lex2(LB, j1) + j2] = fma2_ru(w, C[lex3(LB, j1, j2) + j3], q[lex2(LB, j1) + j2]);
    }
  }
  pair_max<LB>(q, best_l, best_u);
}

// A coefficient pair scaled by the reciprocal bracket sc, both rounded up: l
// is the negated lower coefficient.
__device__ __forceinline__ p2 scale_pair(float l, float u, float2 sc) {
  return pack2(__fmul_ru(l, l >= 0.0f ? sc.y : sc.x), __fmul_ru(u, u >= 0.0f ? sc.y : sc.x));
}

// Whether (n, lb) runs the register kernels, and their launcher.
bool enclose_tail_ok(int n, int lb);
cudaError_t launch_enclose_tail(const Launch& L, const Tables& T, int lb, int64_t n_items, int h,
                                const float* pre_up, const float* pre_lo, int64_t ld,
                                const int32_t* nterms, float* lo, float* hi,
                                const EncloseOpts& ro);

}  // namespace bern
