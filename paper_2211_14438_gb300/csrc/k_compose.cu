// a4: Step 3 of Sec. 5.1 (eqs. post_bounds_1/2): compose the ReLU
// polynomial with the neuron's pre-activation bounds,
//
//   post_up(t) = B(s_up(t)),   post_lo(t) = B(s_lo(t)) - eps,
//   s(t) = (pre(t) - lo) / (hi - lo)  in [0,1] on the box,
//
// as polynomials in t over the graded monomial order, truncated at the
// total-degree cap (dropped terms enter the constant as [min(0,c),max(0,c)]).
//
// Rounding.  s~ = fl((pre - lo*[K=0]) * fl(1/(hi-lo))) is formed in
// round-to-nearest; eta = 5u * sum|s~_K| bounds |s~(t) - s(t)| on the box,
// and Lip = sum_j j|a_j|(1+eta)^(j-1) bounds |B'| there, so Lip*eta is added
// to the upper constant and subtracted from the lower one.  The polynomial
// B(s~(t)) itself is formed with outward rounding:
//   d = 1: c_K = a0[K=0] + a1 s~_K                  (one directed FMA)
//   d = 2: c_K = a0[K=0] + a1 s~_K + a2 (s~^2)_K     (a2 >= 0 by convexity)
// where (s~^2)_K is accumulated round-up for the upper bound and round-down
// for the lower one (a2 >= 0, so each end bounds a2*(s~^2)_K correctly).
//
// Work layout.  A classification kernel puts each item (box, neuron) into a
// queue: zero items only get a term count of 0; identity items and order-1
// items go to an elementwise kernel; order-2 items of input degree D <= 8 go
// to queue D of the squaring kernels (k_compose_square.cu: one lane per item,
// 32 items of equal structure per warp), the rest to a per-item pair-list
// kernel.
#include <algorithm>

#include "compose_common.cuh"

namespace bern {

// ------------------------------------------------------------ classification
// Each block classifies kQueueThreads consecutive items and appends them to the
// queues in item order, reserving its range of every queue with one atomic; so a
// queue is a list of sorted runs, and a warp's 32 consecutive entries are mostly
// neighbouring neurons of one box.
__global__ void __launch_bounds__(kQueueThreads)
k_compose_queue(Tables T, ComposeArgs A, int64_t n_items, int sq_smem, int sq_dmax,
                ComposeScratch S, int* status) {
  const int64_t item = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int q = -1;
  if (item < n_items) {
    const int k = A.kind[item];
    const int Mpre = A.pre_nterms[item];
    int nt = 0;
    if (Mpre < 0 || Mpre > A.pre_cap) {
      atomicOr(status, kStatusInvalid);
    } else if (k == 1) {
      if (Mpre > A.post_ld) {
        atomicOr(status, kStatusCapacity);
      } else {
        q = kQIdent;
        nt = Mpre;
      }
    } else if (k == 2) {
      const int d = A.degrees ? (int)A.degrees[item] : A.global_d;
      const int D = degree_of(T, Mpre);
      if (T.mcount[D] > A.pre_cap || d < 1 || d > kMaxOrder || (A.degrees && d > A.global_d)) {
        atomicOr(status, kStatusInvalid);
      } else {
        const int Mout = T.mcount[min(d * D, A.cap)];
        if (Mout > A.post_ld) {
          atomicOr(status, kStatusCapacity);
        } else if (A.tau > 0.0f || d >= 3) {
          q = d >= kHornerF64Order ? kQHorner64 : kQHorner;
          nt = A.tau > 0.0f ? 0 : Mout;   // with pruning the Horner kernel sets it
        } else if (d == 1) {
          q = kQLinear;
          nt = Mout;
        } else if (D <= sq_smem ||
                   (D <= sq_dmax && !(A.coef[item * kCoefStride + 2] < 0.0f))) {
          q = D;   // past shared memory, a caller's concave polynomial takes the pair lists
          nt = Mout;
        } else if (D <= T.dmax) {
          q = kQPairs;
          nt = Mout;
        } else {
          atomicOr(status, kStatusUnsupported);
        }
      }
    }
    A.post_nterms[item] = nt;
  }
  append_to_lists<kComposeQueues>(q, (int)item, S.qcount, S.queue, S.qcap);
}

// ------------------------------------------------------------ elementwise items
// Identity items copy pre to post: a lane per queue entry (32 consecutive
// entries per warp, so neighbouring lanes touch neighbouring neurons), the
// warps of a block over the coefficient rows.
__global__ void __launch_bounds__(256)
k_compose_copy(ComposeArgs A, ComposeScratch S) {
  const int cnt = S.qcount[kQIdent];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int64_t h = A.h;
  for (int64_t t0 = (int64_t)blockIdx.x * 32; t0 < cnt; t0 += (int64_t)gridDim.x * 32) {
    const int64_t t = t0 + lane;
    if (t >= cnt) continue;
    const int64_t item = S.queue[(int64_t)kQIdent * S.qcap + t];
    const int nt = A.pre_nterms[item];
    const float* su = A.pre_up + A.base(item, A.pre_ld);
    const float* sl = A.pre_lo + A.base(item, A.pre_ld);
    float* du = A.post_up + A.base(item, A.post_ld);
    float* dl = A.post_lo + A.base(item, A.post_ld);
    // four rows of each bound in flight per round
    int r = warp;
    for (; r + 3 * nw < nt; r += 4 * nw) {
      float vu[4], vl[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        vu[q] = su[(r + q * nw) * h];
        vl[q] = sl[(r + q * nw) * h];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        du[(r + q * nw) * h] = vu[q];
        dl[(r + q * nw) * h] = vl[q];
      }
    }
    for (; r < nt; r += nw) {
      du[r * h] = su[r * h];
      dl[r * h] = sl[r * h];
    }
  }
}

// Order-1 items: a_0 + a_1 s~ for both bounds.  A warp takes G entries of the
// queue, lane kl*G + i row kl, kl + 32/G, ... of entry i: eight entries are
// mostly neighbouring neurons, whose rows then come and go in whole sectors.
template <int G>
__device__ __forceinline__ void compose_linear(const ComposeArgs& A, const ComposeScratch& S,
                                               int n_lin, int* status) {
  constexpr int KL = 32 / G;
  const int lane = threadIdx.x & 31;
  const int i = lane % G, kl = lane / G;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  const int64_t h = A.h;
  for (int64_t t = (int64_t)gw * G; t < n_lin; t += (int64_t)nw * G) {
    const bool on = t + i < n_lin;
    const int64_t item = S.queue[(int64_t)kQLinear * S.qcap + (on ? t + i : t)];
    const int Mpre = A.pre_nterms[item];
    const int64_t src = A.base(item, A.pre_ld), dst = A.base(item, A.post_ld);
    const float* Pu = A.pre_up + src;
    const float* Pl = A.pre_lo + src;
    float* Qu = A.post_up + dst;
    float* Ql = A.post_lo + dst;
    const float Lo = A.lo[item], Hi = A.hi[item];
    const float inv = 1.0f / (Hi - Lo);
    const float* cf = A.coef + item * kCoefStride;
    const float a0 = cf[0], a1 = cf[1];
    const int Mout = on ? A.post_nterms[item] : 0;   // the graded prefix of Mpre's degree
    float lu = 0.0f, ll = 0.0f, cu0 = 0.0f, cl0 = 0.0f;
    auto row = [&](int r, float vu, float vl) {
      if (r == 0) {
        vu = __fsub_rn(vu, Lo);
        vl = __fsub_rn(vl, Lo);
      }
      vu = __fmul_rn(vu, inv);
      vl = __fmul_rn(vl, inv);
      lu = __fadd_ru(lu, fabsf(vu));
      ll = __fadd_ru(ll, fabsf(vl));
      const float cu = __fmaf_ru(a1, vu, r == 0 ? a0 : 0.0f);
      const float cl = __fmaf_rd(a1, vl, r == 0 ? a0 : 0.0f);
      if (r == 0) {
        cu0 = cu;
        cl0 = cl;
      } else {
        Qu[r * h] = cu;
        Ql[r * h] = cl;
      }
    };
    int r = kl;
    for (; r + 3 * KL < Mout; r += 4 * KL) {   // four rows of both bounds in flight
      float vu[4], vl[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int rr = r + q * KL;
        vu[q] = rr < Mpre ? Pu[rr * h] : 0.0f;
        vl[q] = rr < Mpre ? Pl[rr * h] : 0.0f;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) row(r + q * KL, vu[q], vl[q]);
    }
    for (; r < Mout; r += KL)
      row(r, r < Mpre ? Pu[r * h] : 0.0f, r < Mpre ? Pl[r * h] : 0.0f);
    __syncwarp();
#pragma unroll
    for (int o = G; o < 32; o <<= 1) {
      lu = __fadd_ru(lu, __shfl_xor_sync(0xffffffffu, lu, o));
      ll = __fadd_ru(ll, __shfl_xor_sync(0xffffffffu, ll, o));
    }
    if (on && kl == 0) {
      const float lip = fabsf(a1);
      const float eu = __fmul_ru(5.0f * kU, lu), el = __fmul_ru(5.0f * kU, ll);
      const float vu = __fadd_ru(cu0, __fmul_ru(lip, eu));
      const float vl = __fsub_rd(__fsub_rd(cl0, __fmul_ru(lip, el)), A.eps[item]);
      Qu[0] = vu;
      Ql[0] = vl;
      if (!isfinite(vu) || !isfinite(vl)) atomicOr(status, kStatusNonFinite);
    }
  }
}

// Eight entries a warp once that leaves each scheduler one or more warps (5120
// boxes of [3,64x4,1] with learned orders, the four layers: 23, 29, 49 and 88 us
// at an entry a warp, now 9, 11, 14 and 19 us), one below; calls of fewer
// neurons take a kernel without the other form, whose instructions a call of 20
// neurons waits 1 us for.
template <bool MANY>
__global__ void __launch_bounds__(256)
k_compose_linear(ComposeArgs A, ComposeScratch S, int few, int* status) {
  const int n_lin = S.qcount[kQLinear];
  if (!MANY || n_lin < few)
    compose_linear<1>(A, S, n_lin, status);
  else
    compose_linear<8>(A, S, n_lin, status);
}

// ------------------------------------------------------------ pair-list squaring
// Order-2 items outside the squaring kernels: one block per item, threads over output
// monomials, symmetric pair lists (I <= J, I + J = K) from the host tables.
__global__ void __launch_bounds__(256)
k_compose_pairs(Tables T, ComposeArgs A, ComposeScratch S, int* status) {
  extern __shared__ float smem[];
  __shared__ float red[32];
  __shared__ float c0[2];
  const int count = S.qcount[kQPairs];
  for (int t = blockIdx.x; t < count; t += gridDim.x) {
    const int64_t item = S.queue[(int64_t)kQPairs * S.qcap + t];
    const int Mpre = A.pre_nterms[item];
    const int Dpre = degree_of(T, Mpre);
    const int Mp = T.mcount[Dpre];
    const int Dfull = 2 * Dpre;
    const int Mout = T.mcount[min(Dfull, A.cap)];
    const int Mfull = T.mcount[Dfull];
    const int h = A.h;
    const float* Pu = A.pre_up + A.base(item, A.pre_ld);
    const float* Pl = A.pre_lo + A.base(item, A.pre_ld);
    float* Qu = A.post_up + A.base(item, A.post_ld);
    float* Ql = A.post_lo + A.base(item, A.post_ld);
    const float L = A.lo[item], H = A.hi[item];
    const float inv = 1.0f / (H - L);
    float* su = smem;
    float* sl = smem + A.pre_cap;
    float au = 0.0f, al = 0.0f;
    for (int r = threadIdx.x; r < Mp; r += blockDim.x) {
      float vu = r < Mpre ? Pu[(int64_t)r * h] : 0.0f, vl = r < Mpre ? Pl[(int64_t)r * h] : 0.0f;
      if (r == 0) {
        vu = __fsub_rn(vu, L);
        vl = __fsub_rn(vl, L);
      }
      vu = __fmul_rn(vu, inv);
      vl = __fmul_rn(vl, inv);
      su[r] = vu;
      sl[r] = vl;
      au = __fadd_ru(au, fabsf(vu));
      al = __fadd_ru(al, fabsf(vl));
    }
    au = block_dsum<true>(au, red);
    __syncthreads();
    al = block_dsum<true>(al, red);
    const float eta_u = __fmul_ru(5.0f * kU, au);
    const float eta_l = __fmul_ru(5.0f * kU, al);
    const float* cf = A.coef + item * kCoefStride;
    const float a0 = cf[0], a1 = cf[1], a2 = cf[2];
    const bool a2pos = a2 >= 0.0f;
    const PairTable pt = T.sq[Dpre];
    float remU = 0.0f, remL = 0.0f;
    for (int K = threadIdx.x; K < Mfull; K += blockDim.x) {
      const int p0 = pt.ptr[K], p1 = pt.ptr[K + 1];
      float offU = 0.0f, offL = 0.0f, diagU = 0.0f, diagL = 0.0f;
      for (int p = p0; p < p1; ++p) {
        const uint32_t pr = pt.pairs[p];
        const int i = pr & 0xffff, j = pr >> 16;
        if (i == j) {
          diagU = __fmul_ru(su[i], su[i]);
          diagL = __fmul_rd(sl[i], sl[i]);
        } else {
          offU = __fmaf_ru(su[i], su[j], offU);
          offL = __fmaf_rd(sl[i], sl[j], offL);
        }
      }
      const float sqU = __fadd_ru(diagU, 2.0f * offU);
      const float sqL = __fadd_rd(diagL, 2.0f * offL);
      const float cu = __fmaf_ru(a2, a2pos ? sqU : sqL,
                                 __fmaf_ru(a1, K < Mp ? su[K] : 0.0f, K == 0 ? a0 : 0.0f));
      const float cl = __fmaf_rd(a2, a2pos ? sqL : sqU,
                                 __fmaf_rd(a1, K < Mp ? sl[K] : 0.0f, K == 0 ? a0 : 0.0f));
      if (K == 0) {
        c0[0] = cu;
        c0[1] = cl;
      } else if (K < Mout) {
        Qu[(int64_t)K * h] = cu;
        Ql[(int64_t)K * h] = cl;
      } else {
        remU = __fadd_ru(remU, fmaxf(cu, 0.0f));
        remL = __fadd_rd(remL, fminf(cl, 0.0f));
      }
    }
    __syncthreads();
    remU = block_dsum<true>(remU, red);
    __syncthreads();
    remL = block_dsum<false>(remL, red);
    if (threadIdx.x == 0) {
      const float lipu = __fmaf_ru(2.0f * fabsf(a2), __fadd_ru(1.0f, eta_u), fabsf(a1));
      const float lipl = __fmaf_ru(2.0f * fabsf(a2), __fadd_ru(1.0f, eta_l), fabsf(a1));
      float cu = __fadd_ru(__fadd_ru(c0[0], __fmul_ru(lipu, eta_u)), remU);
      float cl = __fsub_rd(c0[1], __fmul_ru(lipl, eta_l));
      cl = __fadd_rd(__fsub_rd(cl, A.eps[item]), remL);
      Qu[0] = cu;
      Ql[0] = cl;
      if (!isfinite(cu) || !isfinite(cl)) atomicOr(status, kStatusNonFinite);
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------ launcher
cudaError_t launch_compose(const Launch& L, const Tables& T, const ComposeScratch& S,
                           int64_t n_boxes, int h, int cap, float tau, const int8_t* kind,
                           const float* coef, const float* eps, const uint8_t* degrees,
                           int global_d, const float* lo, const float* hi, const float* pre_up,
                           const float* pre_lo, int64_t pre_ld, const int32_t* pre_nterms,
                           float* post_up, float* post_lo, int64_t post_ld,
                           int32_t* post_nterms, int64_t pre_cap) {
  const int64_t n_items = n_boxes * h;
  if (n_items == 0) return cudaSuccess;
  if (pre_cap <= 0) pre_cap = pre_ld;
  if (!(tau >= 0.0f) || n_items > S.qcap || n_items > INT32_MAX || pre_cap > pre_ld)
    return cudaErrorInvalidValue;
  const bool in_place = post_up == pre_up && post_lo == pre_lo;
  if (in_place && post_ld != pre_ld) return cudaErrorInvalidValue;
  ComposeArgs A{cap, tau, h, kind, coef, eps, degrees, global_d, lo, hi, pre_up, pre_lo, pre_ld,
                pre_nterms, post_up, post_lo, post_ld, post_nterms, pre_cap};
  // the largest input degree any item of this call can have
  int Dmax = 0;
  while (Dmax < kMaxTableDegree && num_monomials(T.n, Dmax + 1) >= 0 &&
         num_monomials(T.n, Dmax + 1) <= pre_cap)
    ++Dmax;
  // long inputs take the squaring kernels where the caller gave them a scratch
  const int sq_smem = std::min(std::min(T.sqt_dmax, Dmax), square_smem_degree(T.n));
  const int sq_dmax =
      S.tws ? std::min(std::min(T.sqt_dmax, Dmax), square_max_degree(T.n)) : sq_smem;
  cudaError_t e = cudaMemsetAsync(S.qcount, 0, kComposeQueues * sizeof(int), L.stream);
  if (e != cudaSuccess) return e;
  k_compose_queue<<<(unsigned)((n_items + kQueueThreads - 1) / kQueueThreads), kQueueThreads, 0,
                    L.stream>>>(
      T, A, n_items, sq_smem, sq_dmax, S, L.status);
  ++*L.launches;
  // order-2 items exist only with order 2 somewhere in the plan (with pruning
  // they go to the Horner kernel)
  const bool order2 = tau == 0.0f && (degrees != nullptr || global_d == 2);
  if (order2) {
    e = launch_compose_square(L, T, S, A, n_items, sq_dmax);
    if (e != cudaSuccess) return e;
  }
  if (!in_place) {   // in place, an identity item's outputs are its inputs
    k_compose_copy<<<(unsigned)std::min<int64_t>((n_items + 31) / 32, device_sms(L) * 16), 256, 0,
                     L.stream>>>(A, S);
    ++*L.launches;
  }
  // order-1 items exist only with order 1 somewhere in the plan (with pruning
  // they go to the Horner kernel)
  if (tau == 0.0f && (degrees != nullptr || global_d == 1)) {
    const int few = 32 * device_sms(L);
    auto kern = n_items < few ? k_compose_linear<false> : k_compose_linear<true>;
    kern<<<(unsigned)std::min<int64_t>((n_items + 7) / 8, device_sms(L) * 16), 256, 0, L.stream>>>(
        A, S, few, L.status);
    ++*L.launches;
  }
  // pair-list kernel for order-2 items beyond the squaring kernels, and for concave
  // ones beyond those in shared memory
  if (order2 && Dmax > sq_smem) {
    const size_t psmem = 2 * (size_t)pre_cap * sizeof(float);
    if (psmem > 200 * 1024) return cudaErrorInvalidValue;
    if (psmem > 48 * 1024) {
      e = cudaFuncSetAttribute(k_compose_pairs, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)psmem);
      if (e != cudaSuccess) return e;
    }
    k_compose_pairs<<<(unsigned)std::min<int64_t>(n_items, device_sms(L) * 8), 256, psmem, L.stream>>>(
        T, A, S, L.status);
    ++*L.launches;
  }
  // Horner kernels for orders >= 3, and for every order when pruning
  if (tau > 0.0f || global_d >= 3) {
    e = launch_compose_horner(L, T, S, A, n_items, Dmax);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

}  // namespace bern
