// a2 (Sec. 5.1 Step 1 with Def. 2) for one to three variables at the orders
// whose last two passes fit a thread's registers, and for order 1.
//
// The passes of enclose_impl.cuh run from the last variable to the first, so
// once the digits of the variables above the second are fixed, what is left
// is a polynomial in t_1, t_2 of at most (l+1)(l+2)/2 coefficients: a thread
// holds those in registers and runs the passes of variables 2 and 1 on
// compile-time indices (line_transform's FMAs, in its order, so every
// coefficient is bit for bit that of the grid kernels).  The lower bound is
// the negated upper bound of the negated polynomial (RD(x) = -RU(-x)), so
// one instruction stream serves both.
//
// Bound: FP32 issue.  The grid in shared memory that it replaces cost a
// shared-memory access for every two FMAs; here the only shared-memory traffic
// is the first pass (three variables: (l+1)(l+2)(l+3)/6 loads, mostly
// broadcasts, per (l+1)(l+2)/2 register coefficients), 1 load to 4 FMAs at
// order 8.
#include <string>

#include "enclose_tail.cuh"

namespace bern {

namespace {

// Threads of a block of the three-variable kernel; a block takes as many items
// as give every thread one (item, digit of t_3) task, or one where the items are
// so few that all threads do best to load its coefficients: up to four of them a
// multiprocessor, two from order 7 on, whose one wave of blocks holds no more (order
// 5, 64 items 4.5 us in full blocks, 3.2 in blocks of their own; 1024 items 4.6 and
// 4.9; order 8, 600 items 5.8 and 6.9).
constexpr int kTailThreads = 128;
template <int LB>
constexpr int tail_items() {
  return kTailThreads / (LB + 1);
}

// Three variables: the scaled coefficients of the block's items sit in shared
// memory in lexicographic order (rows of t_3), a thread takes one digit i_3
// of one item's two polynomials.
template <int LB, int IB>
__global__ void __launch_bounds__(kTailThreads, (LB >= 7 ? 4 : (LB >= 5 ? 6 : 8)))
k_enclose_tail3(Tables T, const float2* __restrict__ rs, int64_t n_items, int h,
                const float* __restrict__ pre_up, const float* __restrict__ pre_lo, int64_t ld,
                const int32_t* __restrict__ nterms, float* __restrict__ lo,
                float* __restrict__ hi, EncloseOpts ro, int* status) {
  constexpr int R = LB + 1, M3 = R * (R + 1) * (R + 2) / 6, MS = M3 | 1;
  constexpr int RB = kTailThreads / IB;                        // rows loaded at a time
  __shared__ p2 s_c[IB * MS];
  __shared__ p2 s_bin[R * R];
  __shared__ float2 s_sc[M3];
  __shared__ int s_at[M3];                     // graded rank -> lexicographic position
  __shared__ int s_bl[IB], s_bu[IB];
  __shared__ float s_rl[IB], s_ru[IB];
  __shared__ int64_t s_item[IB], s_base[IB];
  __shared__ int s_nt[IB], s_any;
  __shared__ p2 s_part[kTailThreads];
  const int tid = threadIdx.x;
  for (int x = tid; x < R * R; x += kTailThreads)
    s_bin[x] = pack2(binomf(x / R, x % R), binomf(x / R, x % R));
  for (int r = tid; r < M3; r += kTailThreads) {
    const int g = __ldg(T.gidx[LB] + r), j1 = g / (R * R), j2 = g / R % R;
    s_at[r] = lex3(LB, j1, j2) + g % R;
    s_sc[r] = __ldg(rs + r);
  }
  const int my = tid % IB, my_r = tid / IB;    // this thread's item and first row in loads
  const int64_t n_list = ro.list ? (int64_t)*ro.count : n_items;
  for (int64_t i0 = (int64_t)blockIdx.x * IB; i0 < n_list; i0 += (int64_t)gridDim.x * IB) {
    __syncthreads();                           // the previous items are finished
    if (tid == 0) s_any = 0;
    if (tid < IB) {
      const int64_t item = i0 + tid < n_list ? (ro.list ? (int64_t)ro.list[i0 + tid] : i0 + tid)
                                             : -1;
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
    if (my_r < RB) {
      // neighbouring threads take neighbouring neurons of one coefficient; all
      // loads of a thread are independent
      const int nt = s_nt[my];
      const float* pu = pre_up + s_base[my];
      const float* pl = pre_lo + s_base[my];
      p2* dst = s_c + my * MS;
#pragma unroll 8
      for (int r = my_r; r < M3; r += RB) {
        const float u = r < nt ? pu[(int64_t)r * h] : 0.0f;
        const float l = r < nt ? -pl[(int64_t)r * h] : 0.0f;
        dst[s_at[r]] = scale_pair(l, u, s_sc[r]);
      }
      if (my_r == 0 && nt > M3) s_any = 1;
    }
    __syncthreads();
    if (s_any)
      remainder_sums<kTailThreads>(pre_up, pre_lo, h, M3, IB, s_base, s_nt, s_part, s_rl, s_ru);
    if (tid < IB * R && i0 + tid / R < n_list) {
      float bl = -CUDART_INF_F, bu = -CUDART_INF_F;
      tail_max<LB>(s_c + tid / R * MS, tid % R, s_bin, bl, bu);
      atomicMax(&s_bl[tid / R], float_key(bl));
      atomicMax(&s_bu[tid / R], float_key(bu));
    }
    __syncthreads();
    if (tid < IB && s_item[tid] >= 0) {
      const int64_t it = s_item[tid];
      const float l = -__fadd_ru(key_float(s_bl[tid]), s_rl[tid]);
      const float u = __fadd_ru(key_float(s_bu[tid]), s_ru[tid]);
      lo[it] = l;
      hi[it] = u;
      if (!(isfinite(l) && isfinite(u))) atomicOr(status, kStatusNonFinite);
      if (ro.kind != nullptr) {
        const int d = ro.degrees ? (int)ro.degrees[it] : ro.global_d;
        ro.kind[it] = (int8_t)relu_item(l, u, d, ro.coef + it * kCoefStride, ro.eps + it, status);
      }
    }
  }
}

// One and two variables: a thread per item, its coefficients straight into registers
// (rank of (j_1, j_2): s (s + 1) / 2 + j_2, s = j_1 + j_2).  Neighbouring
// threads take neighbouring items, each its own terms above the order: at most 150
// rows, and lanes that share them cost calls without any (order 8, 1024 items 5.3
// us for 4.7).
constexpr int kTail2Threads = 128;
template <int NV, int LB>
__global__ void __launch_bounds__(kTail2Threads)
k_enclose_tail2(Tables T, const float2* __restrict__ rs, int64_t n_items, int h,
                const float* __restrict__ pre_up, const float* __restrict__ pre_lo, int64_t ld,
                const int32_t* __restrict__ nterms, float* __restrict__ lo,
                float* __restrict__ hi, EncloseOpts ro, int* status) {
  constexpr int R = LB + 1, M2 = NV == 1 ? R : R * (R + 1) / 2;
  const int64_t n_list = ro.list ? (int64_t)*ro.count : n_items;
  for (int64_t at_list = (int64_t)blockIdx.x * kTail2Threads + threadIdx.x; at_list < n_list;
       at_list += (int64_t)gridDim.x * kTail2Threads) {
    const int64_t item = ro.list ? (int64_t)ro.list[at_list] : at_list;
    int nt = nterms[item];
    if (nt < 0 || nt > ld || nt > T.mexps) {
      atomicOr(status, kStatusInvalid);
      nt = 0;
    }
    const int64_t b = item / h;
    const int64_t base = (b * ld) * h + (item - b * h);
    const float* pu = pre_up + base;
    const float* pl = pre_lo + base;
    // rank r of degree s, exponent j of t_2
    p2 q[M2];
    auto at = [](int s, int j) { return NV == 1 ? s : lex2(LB, s - j) + j; };
#pragma unroll
    for (int s = 0; s <= LB; ++s)
#pragma unroll
      for (int j = 0; j <= (NV == 1 ? 0 : s); ++j) {
        const int r = NV == 1 ? s : s * (s + 1) / 2 + j;
        q[at(s, j)] = r < nt ? pack2(-pl[(int64_t)r * h], pu[(int64_t)r * h]) : pack2(0.0f, 0.0f);
      }
#pragma unroll
    for (int s = 0; s <= LB; ++s)
#pragma unroll
      for (int j = 0; j <= (NV == 1 ? 0 : s); ++j) {
        float l, u;
        unpack2(q[at(s, j)], l, u);
        q[at(s, j)] = scale_pair(l, u, __ldg(rs + (NV == 1 ? s : s * (s + 1) / 2 + j)));
      }
    float bl = -CUDART_INF_F, bu = -CUDART_INF_F;
    if constexpr (NV == 1) {
      pair_transform<LB>(q);
#pragma unroll
      for (int i = 0; i < R; ++i) {
        float l, u;
        unpack2(q[i], l, u);
        bl = fmaxf(bl, l);
        bu = fmaxf(bu, u);
      }
    } else {
      pair_max<LB>(q, bl, bu);
    }
    float ru = 0.0f, rl = 0.0f;
    if (nt > M2) unpack2(thread_remainder(pu, pl, h, M2, nt), rl, ru);
    const float l = -__fadd_ru(bl, rl), u = __fadd_ru(bu, ru);
    lo[item] = l;
    hi[item] = u;
    if (!(isfinite(l) && isfinite(u))) atomicOr(status, kStatusNonFinite);
    if (ro.kind != nullptr) {
      const int d = ro.degrees ? (int)ro.degrees[item] : ro.global_d;
      ro.kind[item] = (int8_t)relu_item(l, u, d, ro.coef + item * kCoefStride, ro.eps + item,
                                        status);
    }
  }
}

// Order 1: the coefficients are the values at the vertices, and with the
// passes' rounding from the last variable to the first the largest is
// a_0 plus the positive linear coefficients in that order.  A thread per
// item, 32 to a warp; SPLIT: iw to a warp, whose lanes share the terms above the
// order.
constexpr int kOrder1Threads = 256;
template <bool SPLIT>
__global__ void __launch_bounds__(kOrder1Threads)
k_enclose_order1(Tables T, int64_t n_items, int h, const float* __restrict__ pre_up,
                 const float* __restrict__ pre_lo, int64_t ld,
                 const int32_t* __restrict__ nterms, float* __restrict__ lo,
                 float* __restrict__ hi, EncloseOpts ro, int iw, int* status) {
  const int n = T.n;
  const int64_t n_list = ro.list ? (int64_t)*ro.count : n_items;
  // SPLIT: warp-uniform, lane 0's item
  const int per = SPLIT ? iw * (kOrder1Threads / 32) : kOrder1Threads;
  const int lane = threadIdx.x & 31;
  for (int64_t i0 = (int64_t)blockIdx.x * per + (SPLIT ? (int)(threadIdx.x >> 5) * iw : threadIdx.x);
       i0 < n_list; i0 += (int64_t)gridDim.x * per) {
    const int64_t at = SPLIT ? i0 + lane : i0;
    const bool mine = !SPLIT || (lane < iw && at < n_list);
    const int64_t item = !mine ? 0 : ro.list ? (int64_t)ro.list[at] : at;
    int nt = mine ? nterms[item] : 0;
    if (nt < 0 || nt > ld || nt > T.mexps) {
      atomicOr(status, kStatusInvalid);
      nt = 0;
    }
    const int64_t b = item / h;
    const int64_t base = (b * ld) * h + (item - b * h);
    float u = 0.0f, l = 0.0f;
    if (nt > 0) {
      u = pre_up[base];
      l = pre_lo[base];
    }
    float cu[kMaxVars], cl[kMaxVars];
#pragma unroll
    for (int k = 0; k < kMaxVars; ++k) {   // rank 1 + k: t_(k+1)
      const bool live = k < n && 1 + k < nt;
      cu[k] = live ? pre_up[base + (int64_t)(1 + k) * h] : 0.0f;
      cl[k] = live ? pre_lo[base + (int64_t)(1 + k) * h] : 0.0f;
    }
#pragma unroll
    for (int k = kMaxVars - 1; k >= 0; --k) {
      u = __fadd_ru(u, fmaxf(cu[k], 0.0f));
      l = __fadd_rd(l, fminf(cl[k], 0.0f));
    }
    float ru = 0.0f, rl = 0.0f;                      // rl: negated
    if constexpr (SPLIT) {
      if (__any_sync(0xffffffffu, nt > n + 1))
        unpack2(warp_remainder(pre_up, pre_lo, h, n + 1, iw, base, nt), rl, ru);
      if (!mine) continue;
    } else {
      if (nt > n + 1) unpack2(thread_remainder(pre_up + base, pre_lo + base, h, n + 1, nt), rl, ru);
    }
    u = __fadd_ru(u, ru);
    l = __fsub_rd(l, rl);
    lo[item] = l;
    hi[item] = u;
    if (!(isfinite(l) && isfinite(u))) atomicOr(status, kStatusNonFinite);
    if (ro.kind != nullptr) {
      const int d = ro.degrees ? (int)ro.degrees[item] : ro.global_d;
      ro.kind[item] = (int8_t)relu_item(l, u, d, ro.coef + item * kCoefStride, ro.eps + item,
                                        status);
    }
  }
}

}  // namespace

bool enclose_tail_ok(int n, int lb) {
  return lb == 1 || (n <= 3 && lb >= 2 && lb <= kTailMaxOrder);
}

cudaError_t launch_enclose_tail(const Launch& L, const Tables& T, int lb, int64_t n_items, int h,
                                const float* pre_up, const float* pre_lo, int64_t ld,
                                const int32_t* nterms, float* lo, float* hi,
                                const EncloseOpts& ro) {
  const int64_t sms = device_sms(L);
  ++*L.launches;
  if (lb == 1) {
    // Fewer items a warp where rows past the order call for more lanes an item and
    // the items do not give eight warps a multiprocessor
    int iw = 32;
    while (iw > 1 && ld > T.n + 1 + 64 && n_items < 8 * sms * iw) iw >>= 1;
    const int64_t per = iw * (kOrder1Threads / 32);
    const int64_t blocks = std::min<int64_t>((n_items + per - 1) / per, sms * 8);
    auto kern = iw < 32 ? k_enclose_order1<true> : k_enclose_order1<false>;
    kern<<<(unsigned)blocks, kOrder1Threads, 0, L.stream>>>(T, n_items, h, pre_up, pre_lo, ld,
                                                            nterms, lo, hi, ro, iw, L.status);
    return cudaGetLastError();
  }
  if (T.n <= 2) {
    const int64_t blocks =
        std::min<int64_t>((n_items + kTail2Threads - 1) / kTail2Threads, sms * 16);
#define BERN_T2(X)                                                                              \
  case X: {                                                                                     \
    auto kern = T.n == 1 ? k_enclose_tail2<1, X> : k_enclose_tail2<2, X>;                       \
    kern<<<(unsigned)blocks, kTail2Threads, 0, L.stream>>>(T, T.rscale[X], n_items, h, pre_up,   \
                                                           pre_lo, ld, nterms, lo, hi, ro, L.status); \
    return cudaGetLastError();                                                                  \
  }
    switch (lb) {
      BERN_T2(2) BERN_T2(3) BERN_T2(4) BERN_T2(5) BERN_T2(6) BERN_T2(7) BERN_T2(8)
      default: return cudaErrorInvalidValue;
    }
#undef BERN_T2
  }
  const bool few = n_items <= (lb <= 6 ? 4 : 2) * sms;
#define BERN_T3(X)                                                                              \
  case X: {                                                                                     \
    const int64_t ib = few ? 1 : tail_items<X>(), need = (n_items + ib - 1) / ib;               \
    auto kern = few ? k_enclose_tail3<X, 1> : k_enclose_tail3<X, tail_items<X>()>;              \
    kern<<<(unsigned)std::min<int64_t>(need, sms * 16), kTailThreads, 0, L.stream>>>(           \
        T, T.rscale[X], n_items, h, pre_up, pre_lo, ld, nterms, lo, hi, ro, L.status);          \
    return cudaGetLastError();                                                                  \
  }
  switch (lb) {
    BERN_T3(2) BERN_T3(3) BERN_T3(4) BERN_T3(5) BERN_T3(6) BERN_T3(7) BERN_T3(8)
    default: return cudaErrorInvalidValue;
  }
#undef BERN_T3
}

}  // namespace bern
