// The last two passes of the Bernstein enclosure in a thread's registers,
// shared by the two- and three-variable kernels (k_enclose_tail.cu) and the
// slab kernel of four and more variables (k_enclose_slab.cu).  Values are
// pairs (negated lower, upper polynomial), packed.cuh.
#pragma once

#include "enclose_impl.cuh"
#include "packed.cuh"

namespace bern {

// Largest order of the register passes of two and three variables: 45 pairs
// of coefficients at order 8 (55 at order 9, the slab kernel's largest).
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

// The terms above the order (ranks `first` on), each in [min(0, a), max(0, a)] on
// the box: the sums of the upper ends and of the negated lower ends, rounded up, as
// (negated lower, upper).  pu, pl: an item's coefficients, of which this thread adds
// every step-th, eight in flight.
//
// Bound: the loads.  One at a time by a thread per item, or by lanes that read a
// neuron's rows at a stride, order 2 on 3003 terms of six variables took 91 us for
// 64 items (11 us now), on degree 16 in three variables 362 us for 32,768 (66).
__device__ __forceinline__ p2 sum_remainder(const float* __restrict__ pu,
                                            const float* __restrict__ pl, int h, int first,
                                            int step, int nt) {
  float ru = 0.0f, rl = 0.0f;
  for (int r = first; r < nt; r += 8 * step) {
    float u[8], l[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int k = r + q * step;
      u[q] = k < nt ? pu[(int64_t)k * h] : 0.0f;
      l[q] = k < nt ? pl[(int64_t)k * h] : 0.0f;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      ru = __fadd_ru(ru, fmaxf(u[q], 0.0f));
      rl = __fadd_ru(rl, fmaxf(-l[q], 0.0f));
    }
  }
  return pack2(rl, ru);
}

// The forms below are out of line: the kernels of 2 to 5 us also wait for their
// instructions, and most calls have no such terms.
//
// Of one item by its thread.
__device__ __noinline__ inline p2 thread_remainder(const float* __restrict__ pu,
                                                   const float* __restrict__ pl, int h, int first,
                                                   int nt) {
  return sum_remainder(pu, pl, h, first, 1, nt);
}

// Of the items of a warp's first iw lanes (a power of two; base and nt theirs): that
// of item lane % iw, its rows split over 32 / iw lanes.
__device__ __noinline__ inline p2 warp_remainder(const float* __restrict__ pre_up,
                                                 const float* __restrict__ pre_lo, int h,
                                                 int first, int iw, int64_t base, int nt) {
  const int lane = threadIdx.x & 31, my = lane & (iw - 1);
  base = __shfl_sync(0xffffffffu, base, my);
  nt = __shfl_sync(0xffffffffu, nt, my);
  p2 v = sum_remainder(pre_up + base, pre_lo + base, h, first + lane / iw, 32 / iw, nt);
  for (int o = iw; o < 32; o <<= 1) v = add2_ru(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Of a block's `ib` items (s_base, s_nt: block and term count of each) into s_rl and
// s_ru.  Called by all NT threads of the block, thread my_r * ib + my on item `my`;
// neighbouring threads read neighbouring neurons of one row, and the item's NT / ib
// partial sums are added in halves.
template <int NT>
__device__ __noinline__ void remainder_sums(const float* __restrict__ pre_up,
                                            const float* __restrict__ pre_lo, int h, int first,
                                            int ib, const int64_t* s_base, const int* s_nt,
                                            p2* s_part, float* s_rl, float* s_ru) {
  const int tid = threadIdx.x, my = tid % ib, my_r = tid / ib, rb = NT / ib;
  p2 v = 0ull;
  if (my_r < rb)
    v = sum_remainder(pre_up + s_base[my], pre_lo + s_base[my], h, first + my_r, rb, s_nt[my]);
  s_part[tid] = v;
  __syncthreads();
  int half = 1;
  while (half < rb) half <<= 1;
  for (half >>= 1; half > 0; half >>= 1) {
    if (my_r < half && my_r + half < rb)
      s_part[tid] = add2_ru(s_part[tid], s_part[tid + half * ib]);
    __syncthreads();
  }
  if (tid < ib) unpack2(s_part[tid], s_rl[tid], s_ru[tid]);
}

// Whether (n, lb) runs the register kernels, and their launcher.
bool enclose_tail_ok(int n, int lb);
cudaError_t launch_enclose_tail(const Launch& L, const Tables& T, int lb, int64_t n_items, int h,
                                const float* pre_up, const float* pre_lo, int64_t ld,
                                const int32_t* nterms, float* lo, float* hi,
                                const EncloseOpts& ro);

}  // namespace bern
