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
// at most 2^-23 of a partial sum that sum |w c| bounds) twice over, and four times
// where a coefficient is positive.  A
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
// a digit at order 8 are packed FMAs; the FP32 pipe is 48% busy).
//
// Order 10 stays on the grids: its 66 pairs of coefficients do not fit a thread's
// registers beside the passes (four variables, 32,768 items 7.2 ms for 2.6 ms, five
// 36 for 26 ms; order 9 1.56 for 1.65 and 6.3 for 19.2 ms).
//
// Three forms, by what fits where (launch_enclose_slab): order 2, and orders 3
// and 4 of few variables, fix every digit above t_3 in registers
// (k_enclose_regs); up to the shared memory of half an SM all slabs of a
// level are made at once, without bounds (k_enclose_expand); above, digit by
// digit with pruning (k_enclose_slab).  Measured against the grid kernels on
// the layers of the [6,100x3,2] network, 2048 boxes: order 2 344 -> 85 us,
// order 4 31.5 -> 1.82 ms (slabs: 3.35 ms), order 8 17.1 -> 2.15 ms.
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
__global__ void __launch_bounds__(NT, NT == 256 ? (LB >= 9 ? 1 : 2) : (NT == 128 ? 5 : 12))
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
  const int per_sm = std::max(1, std::min(NT == 256 ? 2 : (NT == 128 ? 5 : 12), by_smem));
  const int64_t blocks = std::min<int64_t>((int64_t)device_sms(L) * per_sm, n_items);
  kern<<<(unsigned)blocks, NT, smem, L.stream>>>(T, X, sh, T.rscale[LB], n_items, h, pre_up,
                                                 pre_lo, ld, nterms, lo, hi, list, count,
                                                 L.status);
  ++*L.launches;
  return cudaGetLastError();
}

// ------------------------------------------------------------ registers
// Order 2 from four variables on, order 3 up to six and order 4 in four: at
// most 84 coefficients, so a thread fixes all digits above t_3 in registers
// (each level by the same FMAs as slab_row) and runs the digits of t_3; no
// level is stored at all.  64,000 items of four variables at order 4: 64 us
// with the levels in shared memory, 27 us here.
template <int M, int LB>
struct LexRows {
  static constexpr int count() {
    int c = 1;
    for (int i = 1; i < M; ++i) c = c * (LB + i) / i;   // C(M-1+LB, M-1)
    return c;
  }
  int off[count() + 1];
  constexpr LexRows() : off() {
    // rows: the exponents of the first M-1 variables, lexicographic; a row of
    // degree d holds LB - d + 1 coefficients
    int e[M] = {};
    int left = LB, at = 0;
    for (int r = 0; r < count(); ++r) {
      off[r] = at;
      at += left + 1;
      int k = M - 2;
      if (left == 0) {
        while (k > 0 && e[k] == 0) --k;
        left += e[k];
        e[k] = 0;
        --k;
      }
      if (k >= 0) {
        ++e[k];
        --left;
      }
    }
    off[count()] = at;
  }
};

// Digit d of the last of M variables: src (M variables) -> dst (M - 1).
template <int M, int LB, class Src>
__device__ __forceinline__ void fix_digit(const Src& src, int d, const p2* bin,
                                          p2 (&dst)[LexRows<M, LB>::count()]) {
  constexpr LexRows<M, LB> t{};
#pragma unroll
  for (int r = 0; r < LexRows<M, LB>::count(); ++r) dst[r] = src[t.off[r]];
#pragma unroll
  for (int j = 1; j <= LB; ++j)
    if (j <= d) {
      const p2 w = bin[d * (LB + 1) + j];
#pragma unroll
      for (int r = 0; r < LexRows<M, LB>::count(); ++r)
        if (t.off[r + 1] - t.off[r] > j) dst[r] = fma2_ru(w, src[t.off[r] + j], dst[r]);
    }
}

// The largest coefficients over the digits of t_3 of three-variable slab q.
template <int LB>
__device__ __forceinline__ void slab_max(const p2 (&q)[LexRows<4, LB>::count()], float& bl,
                                         float& bu) {
  constexpr LexRows<3, LB> t{};
#pragma unroll
  for (int i3 = 0; i3 <= LB; ++i3) {
    p2 x[LexRows<3, LB>::count()];
#pragma unroll
    for (int r = 0; r < LexRows<3, LB>::count(); ++r) {
      p2 acc = q[t.off[r]];
#pragma unroll
      for (int j = 1; j <= LB; ++j)
        if (j <= i3 && j < t.off[r + 1] - t.off[r])
          acc = i3 == j ? add2_ru(q[t.off[r] + j], acc)
                        : fma2_ru(pack2(cbin(i3, j), cbin(i3, j)), q[t.off[r] + j], acc);
      x[r] = acc;
    }
    pair_max<LB>(x, bl, bu);
  }
}

// The digits of t_M .. t_4 in mixed radix from `digits`, then t_3 .. t_1.
template <int M, int LB, class Src>
__device__ __forceinline__ void fix_all(const Src& src, int digits, const p2* bin, float& bl,
                                        float& bu) {
  p2 dst[LexRows<M, LB>::count()];
  fix_digit<M, LB>(src, digits % (LB + 1), bin, dst);
  if constexpr (M > 4)
    fix_all<M - 1, LB>(dst, digits / (LB + 1), bin, bl, bu);
  else
    slab_max<LB>(dst, bl, bu);
}

constexpr int kRegThreads = 128;
template <int N, int LB>
__global__ void __launch_bounds__(kRegThreads, N >= 8 || LB >= 3 ? 4 : 5)
k_enclose_regs(Tables T, LexView X, const float2* __restrict__ rs, int64_t n_items, int h,
               const float* __restrict__ pre_up, const float* __restrict__ pre_lo, int64_t ld,
               const int32_t* __restrict__ nterms, float* __restrict__ lo, float* __restrict__ hi,
               const int* list, const int* count, int ib, int* status) {
  constexpr int R = LB + 1, MN = LexRows<N + 1, LB>::count(), MS = MN | 1;
  constexpr int TASKS = cipow(R, N - 3);                      // per item
  constexpr int IB = TASKS < kRegThreads ? kRegThreads / TASKS : 1;
  constexpr int RB = kRegThreads / IB;
  __shared__ p2 s_c[IB * MS];
  __shared__ p2 s_bin[R * R];
  __shared__ float2 s_sc[MN];
  __shared__ int s_at[MN];
  __shared__ int s_bl[IB], s_bu[IB];
  __shared__ float s_rl[IB], s_ru[IB];
  __shared__ int64_t s_item[IB], s_base[IB];
  __shared__ int s_nt[IB];
  __shared__ p2 s_part[kRegThreads];
  const int tid = threadIdx.x;
  for (int x = tid; x < R * R; x += kRegThreads)
    s_bin[x] = pack2(binomf(x / R, x % R), binomf(x / R, x % R));
  for (int r = tid; r < MN; r += kRegThreads) {
    s_at[r] = (int)(__ldg(X.pos + r) & 0xffffffu);
    s_sc[r] = __ldg(rs + r);
  }
  const int my = tid % IB, my_r = tid / IB;
  const int64_t n_list = list ? (int64_t)*count : n_items;
  for (int64_t i0 = (int64_t)blockIdx.x * ib; i0 < n_list; i0 += (int64_t)gridDim.x * ib) {
    __syncthreads();                                 // the previous items are finished
    bool above = false;
    if (tid < IB) {
      const bool mine = tid < ib && i0 + tid < n_list;
      const int64_t item = !mine ? -1 : list ? (int64_t)list[i0 + tid] : i0 + tid;
      int nt = item >= 0 ? nterms[item] : 0;
      if (nt < 0 || nt > ld || nt > T.mexps) {
        atomicOr(status, kStatusInvalid);
        nt = 0;
      }
      const int64_t b = item >= 0 ? item / h : 0;
      s_item[tid] = item;
      s_base[tid] = item >= 0 ? (b * ld) * h + (item - b * h) : 0;
      s_nt[tid] = nt;
      s_bl[tid] = float_key(-CUDART_INF_F);
      s_bu[tid] = float_key(-CUDART_INF_F);
      s_rl[tid] = 0.0f;
      s_ru[tid] = 0.0f;
      above = nt > MN;
    }
    if (__syncthreads_or(above))
      remainder_sums<kRegThreads>(pre_up, pre_lo, h, MN, ib, s_base, s_nt, s_part, s_rl, s_ru);
    if (my_r < RB) {
      const int nt = s_nt[my];
      const float* pu = pre_up + s_base[my];
      const float* pl = pre_lo + s_base[my];
#pragma unroll 4
      for (int r = my_r; r < MN; r += RB) {
        const float u = r < nt ? pu[(int64_t)r * h] : 0.0f;
        const float l = r < nt ? -pl[(int64_t)r * h] : 0.0f;
        s_c[my * MS + s_at[r]] = scale_pair(l, u, s_sc[r]);
      }
    }
    __syncthreads();
    for (int t = tid; t < IB * TASKS; t += kRegThreads) {
      const int i = t / TASKS;
      if (i >= ib || i0 + i >= n_list) break;
      float bl = -CUDART_INF_F, bu = -CUDART_INF_F;
      const p2* src = s_c + i * MS;
      fix_all<N, LB>(src, t - i * TASKS, s_bin, bl, bu);
      atomicMax(&s_bl[i], float_key(bl));
      atomicMax(&s_bu[i], float_key(bu));
    }
    __syncthreads();
    if (tid < IB && s_item[tid] >= 0) {
      const int64_t it = s_item[tid];
      const float l = -__fadd_ru(key_float(s_bl[tid]), s_rl[tid]);
      const float u = __fadd_ru(key_float(s_bu[tid]), s_ru[tid]);
      lo[it] = l;
      hi[it] = u;
      if (!(isfinite(l) && isfinite(u))) atomicOr(status, kStatusNonFinite);
    }
  }
}

template <int N, int LB>
cudaError_t launch_regs(const Launch& L, const Tables& T, const LexView& X, int64_t n_items, int h,
                        const float* pre_up, const float* pre_lo, int64_t ld,
                        const int32_t* nterms, float* lo, float* hi, const int* list,
                        const int* count) {
  constexpr int TASKS = cipow(LB + 1, N - 3);
  constexpr int IB = TASKS < kRegThreads ? kRegThreads / TASKS : 1;
  // Items of a block: no more than give every multiprocessor one where rows past the
  // order want all of a block's threads (order 2 on degree 8 in four variables, 64
  // items, 10.2 us in full blocks, 4.4 spread)
  const int64_t sms = device_sms(L);
  const int ib = ld > LexRows<N + 1, LB>::count() + 64
                     ? (int)std::min<int64_t>(IB, std::max<int64_t>(1, n_items / sms)) : IB;
  const int64_t blocks = std::min<int64_t>((n_items + ib - 1) / ib, sms * 16);
  k_enclose_regs<N, LB><<<(unsigned)blocks, kRegThreads, 0, L.stream>>>(
      T, X, T.rscale[LB], n_items, h, pre_up, pre_lo, ld, nterms, lo, hi, list, count, ib,
      L.status);
  ++*L.launches;
  return cudaGetLastError();
}

// ------------------------------------------------------------ expansion
// The same levels without pruning, all slabs of a level at once and several
// items per block, for the shapes whose last level fits shared memory: small
// grids have too few slabs per item to fill a block, and too little behind a
// slab to pay for its bound.
constexpr int64_t kExpandBytes = 52 * 1024;   // shared memory of a block: four per SM
// Of a block with one item: two per SM.  Digit by digit, a small item is a chain of
// barriers (order 3 in eight variables, one item 99 us on the grid, 232 us in slabs,
// 12 us here, 32,768 items 36, 3.6 and 1.2 ms).
constexpr int64_t kExpandOneBytes = 110 * 1024;

struct ExpandShape {
  int n, ib;                   // items per block
  int M[kMaxVars + 1];
  int stride[kMaxVars + 1];    // pairs between the slabs of a level
  int off_tab[kMaxVars + 1];   // row offsets of level m (uint16) in the table area
  int slabs;                   // slabs of the last level per item, R^(n - BOT)
  int off_a, off_b;            // the two level buffers (pairs)
  int total;
};

// BOT: the variables of the last level: three, whose digits run tail_max, or
// four up to order 4, where a thread fixes the digit of t_4 in registers and
// runs all digits of t_3 (fix_all).
template <int LB>
constexpr int expand_bottom() { return LB <= 4 ? 4 : 3; }

template <int LB, int NT>
__global__ void __launch_bounds__(NT, (LB <= 4 ? 4 : 2))
k_enclose_expand(Tables T, LexView X, ExpandShape sh, const float2* __restrict__ rs,
                 int64_t n_items, int h, const float* __restrict__ pre_up,
                 const float* __restrict__ pre_lo, int64_t ld, const int32_t* __restrict__ nterms,
                 float* __restrict__ lo, float* __restrict__ hi, const int* list, const int* count,
                 int* status) {
  constexpr int R = LB + 1, IBMAX = NT / R, BOT = expand_bottom<LB>();
  extern __shared__ p2 sm[];
  __shared__ p2 s_bin[R * R];
  __shared__ int s_bl[IBMAX], s_bu[IBMAX], s_nt[IBMAX], s_any;
  __shared__ float s_rl[IBMAX], s_ru[IBMAX];
  __shared__ int64_t s_item[IBMAX], s_base[IBMAX];
  __shared__ p2 s_part[NT];
  const int tid = threadIdx.x, lane = tid & 31;
  const int n = sh.n, ib = sh.ib, Mn = sh.M[n];
  uint16_t* tab = reinterpret_cast<uint16_t*>(sm);
  for (int x = tid; x < R * R; x += NT) s_bin[x] = pack2(binomf(x / R, x % R), binomf(x / R, x % R));
  for (int m = 4; m <= n; ++m)
    for (int x = tid; x <= sh.M[m - 1]; x += NT)
      tab[sh.off_tab[m] + x] = (uint16_t)__ldg(X.off[m] + x);
  const int my = tid % ib, my_r = tid / ib, rb = NT / ib;
  const int64_t n_list = list ? (int64_t)*count : n_items;
  for (int64_t i0 = (int64_t)blockIdx.x * ib; i0 < n_list; i0 += (int64_t)gridDim.x * ib) {
    __syncthreads();                                 // the previous items are finished
    if (tid == 0) s_any = 0;
    if (tid < ib) {
      const int64_t item = i0 + tid < n_list ? (list ? (int64_t)list[i0 + tid] : i0 + tid) : -1;
      int nt = item >= 0 ? nterms[item] : 0;
      if (nt < 0 || nt > ld || nt > T.mexps) {
        atomicOr(status, kStatusInvalid);
        nt = 0;
      }
      const int64_t b = item >= 0 ? item / h : 0;
      s_item[tid] = item;
      s_base[tid] = item >= 0 ? (b * ld) * h + (item - b * h) : 0;
      s_nt[tid] = nt;
      s_bl[tid] = float_key(-CUDART_INF_F);
      s_bu[tid] = float_key(-CUDART_INF_F);
      s_rl[tid] = 0.0f;
      s_ru[tid] = 0.0f;
    }
    __syncthreads();
    p2* cur = sm + sh.off_a;
    p2* nxt = sm + sh.off_b;
    if (my_r < rb) {
      const int nt = s_nt[my];
      const float* pu = pre_up + s_base[my];
      const float* pl = pre_lo + s_base[my];
      p2* dst = cur + my * sh.stride[n];
#pragma unroll 4
      for (int r = my_r; r < Mn; r += rb) {
        const float u = r < nt ? pu[(int64_t)r * h] : 0.0f;
        const float l = r < nt ? -pl[(int64_t)r * h] : 0.0f;
        dst[__ldg(X.pos + r) & 0xffffffu] = scale_pair(l, u, __ldg(rs + r));
      }
      if (my_r == 0 && nt > Mn) s_any = 1;
    }
    __syncthreads();
    if (s_any)
      remainder_sums<NT>(pre_up, pre_lo, h, Mn, ib, s_base, s_nt, s_part, s_rl, s_ru);
    int ns = ib;                                     // slabs of the level above
    for (int m = n - 1; m >= BOT; --m) {
      const int rows = sh.M[m], sa = sh.stride[m + 1], sb = sh.stride[m];
      const uint16_t* off = tab + sh.off_tab[m + 1];
      const int dq = NT / rows, dr = NT - dq * rows;
      int s = tid / rows, r = tid - s * rows;
      while (s < ns) {
        p2 y[R];
        const int o = off[r];
        slab_row<LB>(cur + s * sa + o, off[r + 1] - o, y);
        p2* dst = nxt + (s * R) * sb + r;
#pragma unroll
        for (int i = 0; i < R; ++i) dst[i * sb] = y[i];
        s += dq;
        r += dr;
        if (r >= rows) {
          r -= rows;
          ++s;
        }
      }
      __syncthreads();
      p2* t = cur;
      cur = nxt;
      nxt = t;
      ns *= R;
    }
    const int per = sh.slabs * R, tasks = ib * per;
    for (int t0 = 0; t0 < tasks; t0 += NT) {
      const int t = t0 + tid;
      const int i = t < tasks ? t / per : -1;
      float bl = -CUDART_INF_F, bu = -CUDART_INF_F;
      if (t < tasks) {
        const p2* slab = cur + t / R * sh.stride[BOT];
        if constexpr (BOT == 4)
          fix_all<4, LB>(slab, t % R, s_bin, bl, bu);
        else
          tail_max<LB>(slab, t % R, s_bin, bl, bu);
      }
      // one update per warp where its lanes share an item
      const int i_first = __shfl_sync(0xffffffffu, i, 0);
      if (__all_sync(0xffffffffu, i == i_first || i < 0)) {
        const int kl = __reduce_max_sync(0xffffffffu, float_key(bl));
        const int ku = __reduce_max_sync(0xffffffffu, float_key(bu));
        if (lane == 0 && i >= 0) {
          atomicMax(&s_bl[i], kl);
          atomicMax(&s_bu[i], ku);
        }
      } else if (i >= 0) {
        atomicMax(&s_bl[i], float_key(bl));
        atomicMax(&s_bu[i], float_key(bu));
      }
    }
    __syncthreads();
    if (tid < ib && s_item[tid] >= 0) {
      const int64_t it = s_item[tid];
      const float l = -__fadd_ru(key_float(s_bl[tid]), s_rl[tid]);
      const float u = __fadd_ru(key_float(s_bu[tid]), s_ru[tid]);
      lo[it] = l;
      hi[it] = u;
      if (!(isfinite(l) && isfinite(u))) atomicOr(status, kStatusNonFinite);
    }
  }
}

// Items per block and shared memory; false where one item does not fit.
template <int LB, int NT>
bool expand_shape(int n, ExpandShape* s) {
  constexpr int R = LB + 1, BOT = expand_bottom<LB>();
  s->n = n;
  int64_t tab = 0;
  for (int m = 0; m <= kMaxVars; ++m) {
    s->M[m] = m == 0 || m > n ? 1 : (int)num_monomials(m, LB);
    s->stride[m] = s->M[m] | 1;
    s->off_tab[m] = (int)tab;
    if (m >= 4 && m <= n) tab += s->M[m - 1] + 1;
  }
  tab = (tab + 3) / 4;                               // pairs
  if (s->M[n] > 65535) return false;
  int64_t a = 0, b = 0, slabs = 1;                   // pairs per item: levels n, n-2, ..; n-1, n-3, ..
  for (int m = n; m >= BOT; --m) {
    int64_t& x = (n - m) & 1 ? b : a;
    x = std::max<int64_t>(x, slabs * s->stride[m]);
    if (m > BOT) slabs *= R;
    if (slabs > 4096) return false;
  }
  s->slabs = (int)slabs;
  int64_t fit = (kExpandBytes / (int64_t)sizeof(p2) - tab) / (a + b);
  if (fit < 1 && tab + a + b <= kExpandOneBytes / (int64_t)sizeof(p2)) fit = 1;
  if (fit < 1) return false;
  const int64_t fill = std::max<int64_t>(1, NT / (slabs * R));   // items whose tasks fill the block
  s->ib = (int)std::min<int64_t>(fit, fill);
  s->off_a = (int)tab;
  s->off_b = (int)(tab + s->ib * a);
  s->total = (int)(tab + s->ib * (a + b));
  return true;
}

template <int LB, int NT>
cudaError_t launch_expand(const Launch& L, const Tables& T, const LexView& X, const ExpandShape& sh,
                          int64_t n_items, int h, const float* pre_up, const float* pre_lo,
                          int64_t ld, const int32_t* nterms, float* lo, float* hi, const int* list,
                          const int* count) {
  const size_t smem = (size_t)sh.total * sizeof(p2);
  auto kern = k_enclose_expand<LB, NT>;
  if (smem > 40 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
  }
  const int64_t need = (n_items + sh.ib - 1) / sh.ib;
  const int64_t blocks = std::min<int64_t>((int64_t)device_sms(L) * 8, need);
  kern<<<(unsigned)blocks, NT, smem, L.stream>>>(T, X, sh, T.rscale[LB], n_items, h, pre_up,
                                                 pre_lo, ld, nterms, lo, hi, list, count,
                                                 L.status);
  ++*L.launches;
  return cudaGetLastError();
}

}  // namespace

#define BERN_SLAB_CASES                                                                       \
  BERN_SLAB(4, 64) BERN_SLAB(5, 128) BERN_SLAB(6, 256) BERN_SLAB(7, 256) BERN_SLAB(8, 256)    \
  BERN_SLAB(9, 256)

bool enclose_slab_ok(const Tables& T, int lb) {
  if (!T.lex || T.n < 4 || lb < 2 || lb > kSlabMaxOrder || !T.lex[lb].pos) return false;
  SlabShape sh;
  switch (lb) {
    case 2: case 3: return true;   // registers, or the expansion
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
  // orders whose levels fit a thread's registers
#define BERN_REGS(N, X)                                                                        \
  if (T.n == N && lb == X)                                                                     \
    return launch_regs<N, X>(L, T, T.lex[X], n_items, h, pre_up, pre_lo, ld, nterms, lo, hi, list, \
                             count);
  BERN_REGS(4, 2) BERN_REGS(5, 2) BERN_REGS(6, 2) BERN_REGS(7, 2) BERN_REGS(8, 2)
  BERN_REGS(4, 3) BERN_REGS(5, 3) BERN_REGS(6, 3) BERN_REGS(4, 4)
#undef BERN_REGS
  // the expansion where its levels fit; the slabs above
#define BERN_EXPAND(X, NT)                                                                     \
  if (lb == X) {                                                                               \
    ExpandShape es;                                                                            \
    if (expand_shape<X, NT>(T.n, &es))                                                         \
      return launch_expand<X, NT>(L, T, T.lex[X], es, n_items, h, pre_up, pre_lo, ld, nterms,  \
                                  lo, hi, list, count);                                        \
  }
  BERN_EXPAND(3, 128) BERN_EXPAND(4, 128) BERN_EXPAND(5, 128)
  BERN_EXPAND(6, 256) BERN_EXPAND(7, 256) BERN_EXPAND(8, 256)
#undef BERN_EXPAND
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
