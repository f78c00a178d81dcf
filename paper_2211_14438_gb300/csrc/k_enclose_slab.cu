// a2 (Sec. 5.1 Step 1 with Def. 2) for four and more variables at orders
// 2..kSlabMaxOrder: the range of the Bernstein coefficients without the grid.
//
// The passes run from the last variable to the first.  Fixing the digit i of
// the last variable turns a polynomial in m variables into one in m - 1 (the
// "slab" of that digit: C(m-1+l, l) sums of at most l + 1 coefficients); the
// slabs of all digits, taken recursively, hold every line of every pass once,
// with the FMAs of line_transform in its order, so every coefficient is bit
// for bit that of a grid of (l+1)^n cells - but a polynomial of three
// variables (165 coefficients at order 8) is all that has to be kept, not
// 9^6 cells, and the last two passes run in a thread's registers
// (enclose_tail.cuh).  With the polynomial's coefficients in lexicographic
// order every slab reads contiguous rows.
//
// Slabs that cannot hold the extreme are left out.  All weights of the passes
// below a slab are at most C(l, j), so no coefficient in it exceeds
//   c_0 + sum_J max(0, w_J c_J),   w_J = prod_k C(l, j_k),
// and no computed one exceeds that by more than delta sum_J |w_J c_J|, where
// delta covers the roundings of the m remaining passes (m l additions, each of
// at most 2^-23 of a partial sum that sum |w c| bounds) four times over.  A
// slab whose bound is not above the largest coefficient found so far adds
// nothing to the maximum.  The search starts from the value at the vertex that
// the linear terms point to (summed rounding down, so it is not above the
// computed coefficient there).
//
// Work layout: a block of NT threads per item, both bounds at once as pairs
// (negated lower, upper), packed.cuh: RD(x) = -RU(-x), so one instruction
// stream serves both.  A level is made from the rows of the one above: a thread
// loads a row (the coefficients that differ in the last exponent), transforms
// it in registers and stores one value into the slab of every digit.  Levels
// of five and more variables are made one digit at a time, the slabs of four
// and three variables for all digits; then a thread takes a digit of t_3 of a
// three-variable slab and runs the last two passes in registers.
//
// Bound: FP32 issue in the register passes (610 of about 1000 instructions of
// a digit at order 8 are packed FMAs).
#include "enclose_tail.cuh"

namespace bern {

namespace {

struct SlabShape {
  int M[kMaxVars + 1];         // coefficients of m variables
  int n;
  int off_s[kMaxVars + 1];     // shared-memory offsets (pairs) of the levels 5..n-1
  int off_b, off_c;            // four- and three-variable slabs
  int off_w4;                  // weights of four variables (two floats a pair)
  int total;                   // pairs
};

__device__ __forceinline__ p2 warp_sum2(p2 v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = add2_ru(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
template <int NT>
__device__ __forceinline__ p2 block_sum2(p2 v, p2* red) {
  v = warp_sum2(v);
  if constexpr (NT > 32) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    v = lane < NT / 32 ? red[lane] : 0ull;
    v = warp_sum2(v);
  }
  return v;
}

// The part of a slab's bound that one coefficient pair adds, c the coefficient
// and w its weight: max(t, -delta t), t = w c, is at least max(0, t) and, with
// the factor 1 + delta on the sum, covers the rounding share.
__device__ __forceinline__ p2 bound_part(p2 c, float w, float delta) {
  float l, u;
  unpack2(mul2_ru(pack2(w, w), c), l, u);
  return pack2(fmaxf(l, -delta * l), fmaxf(u, -delta * u));
}
// Whether the bound of a slab (constant c0, sum of bound_part over the rest)
// exceeds what was found so far for either polynomial.
__device__ __forceinline__ bool bound_live(p2 c0, p2 sum, float delta, float best_l, float best_u) {
  float cl, cu, l, u;
  unpack2(c0, cl, cu);
  unpack2(sum, l, u);
  const float g = 1.0f + 2.0f * delta;
  l = __fadd_ru(__fadd_ru(cl, __fmul_ru(l, g)), __fmaf_ru(delta, fabsf(cl), 1e-36f));
  u = __fadd_ru(__fadd_ru(cu, __fmul_ru(u, g)), __fmaf_ru(delta, fabsf(cu), 1e-36f));
  return !(l <= best_l && u <= best_u);
}
// The rounding share of a bound over m variables at order l.
__device__ __forceinline__ float slab_delta(int m, int l) { return (float)(m * l + 16) * 0x1p-22f; }

// A warp decides whether the slab c (rows coefficients) is visited.
__device__ __forceinline__ bool warp_live(const p2* c, const float* wt, int rows,
                                          float delta, float best_l, float best_u) {
  const int lane = threadIdx.x & 31;
  p2 sum = 0ull;
  for (int r = lane; r < rows; r += 32)
    if (r > 0) sum = add2_ru(sum, bound_part(c[r], wt[r], delta));
  return bound_live(c[0], warp_sum2(sum), delta, best_l, best_u);
}

// Four-variable slabs taken per inner step, so that the digits of their
// three-variable slabs fill the block.
template <int LB, int NT>
constexpr int slab_group() {
  const int R = LB + 1, g = NT / (R * R);
  return NT <= 64 || g > R ? R : (g < 1 ? 1 : g);
}

// One row of a level in registers: its coefficients transformed in place, y[i]
// the value of digit i.
template <int LB>
__device__ __forceinline__ void slab_row(const p2* __restrict__ src, int len, p2 (&y)[LB + 1]) {
#pragma unroll
  for (int j = 0; j <= LB; ++j) y[j] = j < len ? src[j] : 0ull;
  pair_transform<LB>(y);
}

template <int LB, int NT>
__global__ void __launch_bounds__(NT, NT == 256 ? (LB >= 9 ? 1 : 2) : (NT == 128 ? 5 : (NT == 64 ? 12 : 24)))
k_enclose_slab(Tables T, LexView X, SlabShape sh, const float2* __restrict__ rs, int64_t n_items,
               int h, const float* __restrict__ pre_up, const float* __restrict__ pre_lo,
               int64_t ld, const int32_t* __restrict__ nterms, float* __restrict__ lo,
               float* __restrict__ hi, const int* list, const int* count, int* status) {
  constexpr int R = LB + 1, NW = NT / 32, GB = slab_group<LB, NT>();
  constexpr int M3 = R * (R + 1) * (R + 2) / 6, M3S = M3 | 1;
  extern __shared__ p2 sm[];
  __shared__ p2 s_bin[R * R];
  __shared__ p2 red[32];
  __shared__ uint16_t s_off4[M3 + 1];                // rows of four variables
  __shared__ int s_bl, s_bu, s_live;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = sh.n, M4 = sh.M[4];
  p2* c = sm;
  p2* B = sm + sh.off_b;
  p2* Cs = sm + sh.off_c;
  for (int x = tid; x < R * R; x += NT) s_bin[x] = pack2(binomf(x / R, x % R), binomf(x / R, x % R));
  for (int x = tid; x <= M3; x += NT) s_off4[x] = (uint16_t)__ldg(X.off[4] + x);
  float* w4 = reinterpret_cast<float*>(sm + sh.off_w4);   // five and more variables
  if (n >= 5)
    for (int x = tid; x < M4; x += NT) w4[x] = __ldg(X.wt[4] + x);
  const int64_t n_list = list ? (int64_t)*count : n_items;
  for (int64_t p = blockIdx.x; p < n_list; p += gridDim.x) {
    const int64_t item = list ? (int64_t)list[p] : p;
    int nt = nterms[item];
    if (nt < 0 || nt > ld || nt > T.mexps) {
      if (tid == 0) atomicOr(status, kStatusInvalid);
      nt = 0;
    }
    const int64_t b = item / h;
    const float* pu = pre_up + (b * ld) * h + (item - b * h);
    const float* pl = pre_lo + (b * ld) * h + (item - b * h);
    const int m_eff = T.mcount[min(prefix_degree(T, nt), LB)];
    unsigned Vl = 0, Vu = 0;                         // the vertices of the linear terms
    for (int k = 0; k < n; ++k)
      if (1 + k < nt) {
        if (pl[(int64_t)(1 + k) * h] < 0.0f) Vl |= 1u << k;
        if (pu[(int64_t)(1 + k) * h] > 0.0f) Vu |= 1u << k;
      }
    __syncthreads();                                 // the previous item is finished
    for (int x = nt + tid; x < sh.M[n]; x += NT)     // ranks the item does not hold
      c[__ldg(X.pos + x) & 0xffffffu] = 0ull;
    p2 rem = 0ull, vert = 0ull;                      // vert: negated sums, rounded up
#pragma unroll 4
    for (int r = tid; r < nt; r += NT) {
      const float u = pu[(int64_t)r * h], l = -pl[(int64_t)r * h];
      if (r < m_eff) {
        const uint32_t at = __ldg(X.pos + r);
        c[at & 0xffffffu] = scale_pair(l, u, rs[r]);
        vert = add2_ru(vert, pack2(((at >> 24) & ~Vl) == 0 ? -l : 0.0f,
                                   ((at >> 24) & ~Vu) == 0 ? -u : 0.0f));
      } else {
        rem = add2_ru(rem, pack2(fmaxf(l, 0.0f), fmaxf(u, 0.0f)));
      }
    }
    vert = block_sum2<NT>(vert, red);
    rem = block_sum2<NT>(rem, red);
    if (tid == 0) {
      float vl, vu;
      unpack2(vert, vl, vu);
      s_bl = float_key(isfinite(vl) ? -vl : -CUDART_INF_F);
      s_bu = float_key(isfinite(vu) ? -vu : -CUDART_INF_F);
    }
    __syncthreads();
    // visits the slabs below a five-variable slab (four variables: c itself)
    auto inner = [&](const p2* s5) {
      unsigned live = 1u;                            // the digits of t_5 still to visit
      if (n >= 5) {
        if (tid == 0) s_live = 0;
        const int32_t* off = X.off[5];
        for (int r = tid; r < M4; r += NT) {
          p2 y[R];
          const int o = __ldg(off + r);
          slab_row<LB>(s5 + o, __ldg(off + r + 1) - o, y);
#pragma unroll
          for (int i = 0; i < R; ++i) B[i * M4 + r] = y[i];
        }
        __syncthreads();
        for (int t = warp; t < R; t += NW)
          if (warp_live(B + t * M4, w4, M4, slab_delta(4, LB), key_float(s_bl), key_float(s_bu)) &&
              lane == 0)
            atomicOr(&s_live, 1 << t);
        __syncthreads();
        live = s_live;
      }
      while (live) {
        int ng = 0, grp[GB];
#pragma unroll
        for (int g = 0; g < GB; ++g) {
          grp[g] = 0;
          if (live) {
            grp[g] = __ffs(live) - 1;
            live &= live - 1;
            ++ng;
          }
        }
        for (int x = tid; x < ng * M3; x += NT) {
          const int g = x / M3, r = x - g * M3;
          int src = 0;
#pragma unroll
          for (int k = 0; k < GB; ++k)
            if (g == k) src = grp[k];
          p2 y[R];
          const int o = s_off4[r];
          slab_row<LB>((n >= 5 ? B + src * M4 : c) + o, s_off4[r + 1] - o, y);
#pragma unroll
          for (int i = 0; i < R; ++i) Cs[(g * R + i) * M3S + r] = y[i];
        }
        __syncthreads();
        const int tasks = ng * R * R;
        float bl = -CUDART_INF_F, bu = -CUDART_INF_F;
        for (int t = tid; t < tasks; t += NT) tail_max<LB>(Cs + t / R * M3S, t % R, s_bin, bl, bu);
        bl = warp_max(bl);
        bu = warp_max(bu);
        if (lane == 0) {
          atomicMax(&s_bl, float_key(bl));
          atomicMax(&s_bu, float_key(bu));
        }
        __syncthreads();
      }
    };
    if (n <= 5) {
      inner(c);
    } else {
      // digits of t_n .. t_6, one level of slabs at a time
      int m = n - 1;
      uint64_t dig = 0;                              // 4 bits per level
      for (;;) {
        const int i = (int)(dig >> (4 * m)) & 15;
        const p2* src = m + 1 == n ? c : sm + sh.off_s[m + 1];
        p2* dst = sm + sh.off_s[m];
        const int32_t* off = X.off[m + 1];
        const float* wt = X.wt[m];
        const float delta = slab_delta(m, LB);
        p2 sum = 0ull;
        for (int r = tid; r < sh.M[m]; r += NT) {
          const int o = __ldg(off + r), jm = min(i, __ldg(off + r + 1) - o - 1);
          p2 acc = src[o];
          for (int j = 1; j <= jm; ++j) acc = fma2_ru(s_bin[i * R + j], src[o + j], acc);
          dst[r] = acc;
          if (r > 0) sum = add2_ru(sum, bound_part(acc, __ldg(wt + r), delta));
        }
        sum = block_sum2<NT>(sum, red);
        __syncthreads();                             // dst is complete; the best are settled
        if (bound_live(dst[0], sum, delta, key_float(s_bl), key_float(s_bu))) {   // block-uniform
          if (m == 5) {
            inner(dst);
          } else {
            --m;
            dig &= ~((uint64_t)15 << (4 * m));
            continue;
          }
        }
        while (m < n && ((int)(dig >> (4 * m)) & 15) == LB) ++m;
        if (m == n) break;
        dig += (uint64_t)1 << (4 * m);
        __syncthreads();                             // dst is reused
      }
    }
    __syncthreads();
    if (tid == 0) {
      float rl, ru;
      unpack2(rem, rl, ru);
      const float l = -__fadd_ru(key_float(s_bl), rl), u = __fadd_ru(key_float(s_bu), ru);
      lo[item] = l;
      hi[item] = u;
      if (!(isfinite(l) && isfinite(u))) atomicOr(status, kStatusNonFinite);
    }
  }
}

template <int LB, int NT>
bool shape_of(int n, SlabShape* s) {
  constexpr int R = LB + 1, GB = slab_group<LB, NT>();
  s->n = n;
  for (int m = 0; m <= kMaxVars; ++m) {
    s->off_s[m] = 0;
    s->M[m] = m == 0 || m > n ? 1 : (int)num_monomials(m, LB);
  }
  int64_t off = s->M[n];
  for (int m = n - 1; m >= 5; --m) {
    s->off_s[m] = (int)off;
    off += s->M[m];
  }
  s->off_b = (int)off;
  if (n >= 5) off += (int64_t)R * s->M[4];
  s->off_c = (int)off;
  off += (int64_t)(n >= 5 ? GB : 1) * R * (s->M[3] | 1);
  s->off_w4 = (int)off;
  if (n >= 5) off += (s->M[4] + 1) / 2;
  s->total = (int)off;
  return off * (int64_t)sizeof(p2) <= 220 * 1024;
}

template <int LB, int NT>
cudaError_t launch_slab(const Launch& L, const Tables& T, const LexView& X, int64_t n_items, int h,
                        const float* pre_up, const float* pre_lo, int64_t ld,
                        const int32_t* nterms, float* lo, float* hi, const int* list,
                        const int* count) {
  SlabShape sh;
  if (!shape_of<LB, NT>(T.n, &sh)) return cudaErrorInvalidValue;
  const size_t smem = (size_t)sh.total * sizeof(p2);
  auto kern = k_enclose_slab<LB, NT>;
  if (smem > 47 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
  }
  const int by_smem = (int)((226 * 1024) / (smem + 3072));
  const int per_sm = std::max(1, std::min(NT == 256 ? 2 : (NT == 128 ? 5 : (NT == 64 ? 12 : 24)), by_smem));
  const int64_t blocks = std::min<int64_t>((int64_t)device_sms(L) * per_sm, n_items);
  kern<<<(unsigned)blocks, NT, smem, L.stream>>>(T, X, sh, T.rscale[LB], n_items, h, pre_up,
                                                 pre_lo, ld, nterms, lo, hi, list, count,
                                                 L.status);
  ++*L.launches;
  return cudaGetLastError();
}

}  // namespace

#define BERN_SLAB_CASES                                                                       \
  BERN_SLAB(2, 32) BERN_SLAB(3, 32) BERN_SLAB(4, 64) BERN_SLAB(5, 128) BERN_SLAB(6, 256)      \
  BERN_SLAB(7, 256) BERN_SLAB(8, 256) BERN_SLAB(9, 256) BERN_SLAB(10, 256)

bool enclose_slab_ok(const Tables& T, int lb) {
  if (!T.lex || T.n < 4 || lb < 2 || lb > kSlabMaxOrder || !T.lex[lb].pos) return false;
  SlabShape sh;
  switch (lb) {
#define BERN_SLAB(X, NT) case X: return shape_of<X, NT>(T.n, &sh);
    BERN_SLAB_CASES
#undef BERN_SLAB
    default: return false;
  }
}

cudaError_t launch_enclose_slab(const Launch& L, const Tables& T, int lb, int64_t n_items, int h,
                                const float* pre_up, const float* pre_lo, int64_t ld,
                                const int32_t* nterms, float* lo, float* hi, const int* list,
                                const int* count) {
  switch (lb) {
#define BERN_SLAB(X, NT) \
  case X: return launch_slab<X, NT>(L, T, T.lex[X], n_items, h, pre_up, pre_lo, ld, nterms, lo, hi, \
                                    list, count);
    BERN_SLAB_CASES
#undef BERN_SLAB
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace bern
