// a4 for order-2 items of input degree D <= 8: a0 + a1 s + a2 s^2 of both bounds
// of 32 items per group, one lane per item, every control decision uniform.
//
// The square is a sum over products of parts of s whose exponents of all but
// the last one or two variables agree:
//   * a tile is the part with given exponents of t_1..t_(n-2), a triangle in
//     (t_(n-1), t_n) of degree d; the output tile of prefix Q, degree
//     e = 2D - |Q|, is the sum over the prefix pairs P1 + P2 = Q of the products
//     of their tiles (d1 + d2 = e).  Up to e = kTileDegree its (e+1)(e+2)/2 <=
//     21 accumulator pairs stay in registers and a pair is one block of unrolled
//     FMAs, |T1||T2| of them for |T1| + |T2| loads (e = 6, 28 pairs, spills:
//     3.5 against 3.1 ms on the layer below);
//   * above, one output row of t_n at a time (at most 17 accumulators), from the
//     1-D convolutions of row pairs, up to 9 x 9.
// Both are units of one list, dispatched on the pair's degrees (lengths).  The
// tiles are what makes the products dense where there are many variables: at
// degree 4 in six variables a row pair has 2.8 products on average, a tile
// pair 9.
//
// Both bounds are pairs (packed.cuh), s as (lower, upper), accumulators as
// (negated lower, upper): an off-diagonal pair multiplies -+2 s by s (exact
// scaling), the diagonal pair s by s once, everything rounds up.
//
// s lies in shared memory (32 lanes x M pairs) up to kSquareSmemTerms terms; for
// longer inputs a first kernel writes it to a scratch [M][32] per group (1 MB with
// 3003 terms, up to 512 MB of groups in a pass; some hundred of them stay in the L2),
// and the units of a group are spread over blocks.
//
// Bound: instruction issue (n = 6, D = 4: 22,155 products, 2,575 tile or row
// pairs and 3,003 outputs of both bounds per group; 52% of the issue slots, ALU the
// busiest pipe) and, from degree 8 in three variables, DRAM traffic of partly
// written sectors (the stable neurons between the items): 53% of the measured
// bandwidth.  Against 1-D rows with a launch per bound: layer 3 of [6,100x3,2],
// 2048 boxes, 7.31 -> 2.66 ms; layer 4 of [3,64x4,1], 5120 boxes, 1.28 -> 1.16
// ms.  Against a block per item over pair lists (each thread gathering its own
// list): layer 4 of [6,64x4,1], degree 8, 48 boxes, 51.4 -> 6.4 ms.
#include <algorithm>

#include "compose_common.cuh"
#include "packed.cuh"

namespace bern {

namespace {

constexpr int kRowHalf = kRowLen / 2 + 1;    // pairs of coefficients of the longest row

// Triangles of degree d: row r of t_n has d - r + 1 coefficients.  In the
// accumulators rows follow one another; in the inputs every row is padded with
// zeros to an even length, so that a 16-byte load takes two pairs.
__host__ __device__ constexpr int tri_row(int d, int r) { return r * (d + 1) - r * (r - 1) / 2; }
__host__ __device__ constexpr int tri_size(int d) { return (d + 1) * (d + 2) / 2; }

// s of this lane's item, two coefficients at a time from an even position:
// shared memory or the group's scratch.
struct SmemRow {
  const p2* s;
  __device__ __forceinline__ ulonglong2 two(int i) const {
    return *reinterpret_cast<const ulonglong2*>(s + i);
  }
};
struct ScratchRow {
  const p2* s;                               // [position / 2][lane][2]
  __device__ __forceinline__ ulonglong2 two(int i) const {
    return __ldg(reinterpret_cast<const ulonglong2*>(s + 32 * i));
  }
};

// Row r of a tile of degree D at position o into y.
template <int N, class Row>
__device__ __forceinline__ void load_row(const Row& s, int o, p2* y) {
#pragma unroll
  for (int c = 0; c < N; c += 2) {
    const ulonglong2 v = s.two(o + c);
    y[c] = v.x;
    if (c + 1 < N) y[c + 1] = v.y;
  }
}

// acc += 2 T1 T2 of tiles of degrees D1 <= D2; acc is a triangle of degree D1 + D2
// in registers.  T1 is held, T2 taken a row at a time from the last
// to the first.  So every output coefficient adds its row pairs by rising row of
// T1 and the products of a row pair by rising exponent in the shorter row (in T1
// when equal): the order of the 1-D convolutions over a list of row pairs
// sorted that way, which the fused layer (k_layer.cu) follows bit for bit.
template <int D1, int D2, int R2, class Row>
__device__ __forceinline__ void tile_rows(const Row& s, int o2, const p2 (&x)[tri_size(D1)],
                                          p2 (&acc)[tri_size(D1 + D2)]) {
  constexpr int n2 = D2 - R2 + 1;
  p2 y[n2];
  load_row<n2>(s, o2 + pad_row(D2, R2), y);
#pragma unroll
  for (int r1 = 0; r1 <= D1; ++r1) {
    const int n1 = D1 - r1 + 1;
    if (n1 <= n2) {
#pragma unroll
      for (int c1 = 0; c1 < n1; ++c1)
#pragma unroll
        for (int c2 = 0; c2 < n2; ++c2) {
          p2& a = acc[tri_row(D1 + D2, r1 + R2) + c1 + c2];
          a = fma2_ru(x[tri_row(D1, r1) + c1], y[c2], a);
        }
    } else {
#pragma unroll
      for (int c2 = 0; c2 < n2; ++c2)
#pragma unroll
        for (int c1 = 0; c1 < n1; ++c1) {
          p2& a = acc[tri_row(D1 + D2, r1 + R2) + c1 + c2];
          a = fma2_ru(x[tri_row(D1, r1) + c1], y[c2], a);
        }
    }
  }
  if constexpr (R2 > 0) tile_rows<D1, D2, R2 - 1>(s, o2, x, acc);
}
template <int D, int R, class Row>
__device__ __forceinline__ void load_tile(const Row& s, int o, p2 (&y)[tri_size(D)]) {
  load_row<D - R + 1>(s, o + pad_row(D, R), y + tri_row(D, R));
  if constexpr (R < D) load_tile<D, R + 1>(s, o, y);
}
template <int D1, int D2, class Row>
__device__ __forceinline__ void tile_pair(const Row& s, int o1, int o2,
                                          p2 (&acc)[tri_size(D1 + D2)]) {
  p2 x[tri_size(D1)];
  load_tile<D1, 0>(s, o1, x);
#pragma unroll
  for (int i = 0; i < tri_size(D1); ++i) x[i] = mul2_ru(pack2(-2.0f, 2.0f), x[i]);
  tile_rows<D1, D2, D2>(s, o2, x, acc);
}

// acc += T^2 of a tile of degree D1: its row pairs r1 < r2 (each product counts
// twice), then the rows' own squares, in the same order.
template <int D1, class Row>
__device__ __forceinline__ void tile_diag(const Row& s, int o, p2 (&acc)[tri_size(2 * D1)]) {
  p2 y[tri_size(D1)];
  load_tile<D1, 0>(s, o, y);
#pragma unroll
  for (int r1 = 0; r1 <= D1; ++r1)
#pragma unroll
    for (int r2 = r1; r2 <= D1; ++r2)
#pragma unroll
      for (int c2 = 0; c2 <= D1 - r2; ++c2) {      // row r2: the shorter
        const p2 x = mul2_ru(pack2(-1.0f, 1.0f), y[tri_row(D1, r2) + c2]), x2 = add2_ru(x, x);
#pragma unroll
        for (int c1 = r1 == r2 ? c2 : 0; c1 <= D1 - r1; ++c1) {
          p2& a = acc[tri_row(2 * D1, r1 + r2) + c1 + c2];
          a = fma2_ru(r1 == r2 && c1 == c2 ? x : x2, y[tri_row(D1, r1) + c1], a);
        }
      }
}

// The same for rows of t_n of padded half lengths H1 <= H2 (a padded product adds
// an exact zero): 15 cases instead of one per pair of lengths keep the code
// within the instruction cache.
constexpr int kRowAcc = 4 * kRowHalf;
template <int H1, int H2, class Row>
__device__ __forceinline__ void row_pair(const Row& s, int o1, int o2, p2 (&acc)[kRowAcc]) {
  p2 x[2 * H1], y[2 * H2];
  load_row<2 * H1>(s, o1, x);
  load_row<2 * H2>(s, o2, y);
#pragma unroll
  for (int a = 0; a < 2 * H1; ++a) {
    x[a] = mul2_ru(pack2(-2.0f, 2.0f), x[a]);
#pragma unroll
    for (int b = 0; b < 2 * H2; ++b) acc[a + b] = fma2_ru(x[a], y[b], acc[a + b]);
  }
}
template <int H, class Row>
__device__ __forceinline__ void row_diag(const Row& s, int o, p2 (&acc)[kRowAcc]) {
  p2 y[2 * H];
  load_row<2 * H>(s, o, y);
#pragma unroll
  for (int a = 0; a < 2 * H; ++a) {
    const p2 x = mul2_ru(pack2(-1.0f, 1.0f), y[a]), x2 = add2_ru(x, x);
    acc[2 * a] = fma2_ru(x, y[a], acc[2 * a]);
#pragma unroll
    for (int b = a + 1; b < 2 * H; ++b) acc[a + b] = fma2_ru(x2, y[b], acc[a + b]);
  }
}

#define BERN_RP(A, B) \
  case row_half_case(A, B): row_pair<A, B>(s, o1, o2, acc); break;
#define BERN_ROW_CASES                                                                      \
  BERN_RP(1, 1) BERN_RP(1, 2) BERN_RP(1, 3) BERN_RP(1, 4) BERN_RP(1, 5) BERN_RP(2, 2)       \
  BERN_RP(2, 3) BERN_RP(2, 4) BERN_RP(2, 5) BERN_RP(3, 3) BERN_RP(3, 4) BERN_RP(3, 5)       \
  BERN_RP(4, 4) BERN_RP(4, 5) BERN_RP(5, 5)
#define BERN_RD(A) \
  case A: row_diag<A>(s, o1, acc); break;
static_assert(kRowHalf == 5, "the cases above");

// What a lane needs to write its item's coefficients.
struct SquareOut {
  float* QU;
  float* QL;
  int h;
  p2 a1, a2;                 // (-a1, a1), (a2, a2)
  int Mout;                  // ranks kept under the cap
  bool valid;                // the lane has an item
};

// One output coefficient pair from its square (negated lower, upper) and s:
// written, or (TRUNC: some outputs of the degree exceed the cap) added to the
// remainder.  Returns the value.
template <bool TRUNC>
__device__ __forceinline__ p2 put(const SquareOut& o, p2 sq, p2 lin, int K, p2& rem) {
  const p2 v = fma2_ru(o.a2, sq, mul2_ru(o.a1, lin));
  float vl, vu;
  unpack2(v, vl, vu);
  if (!TRUNC || K < o.Mout) {
    if (o.valid) {
      o.QU[(int64_t)K * o.h] = vu;
      o.QL[(int64_t)K * o.h] = -vl;
    }
  } else {
    rem = add2_ru(rem, pack2(fmaxf(vl, 0.0f), fmaxf(vu, 0.0f)));
  }
  return v;
}

// A unit's header with the first 32 words of its pairs and its output ranks (at
// most 21 of a tile, 17 of a row), one per lane.
struct UnitHead {
  int4 un;
  uint32_t words;
  int32_t rank;
};
static_assert(kTileDegree == 5, "the tiles of square_unit");
static_assert(tri_size(kTileDegree) <= 32 && 2 * kRowLen - 1 <= 32, "a lane per output");
__device__ __forceinline__ UnitHead unit_head(const SquareTable& R, int4 un) {
  const int lane = threadIdx.x & 31;
  UnitHead h;
  h.un = un;
  h.words = un.x + lane < un.y ? __ldg(R.words + un.x + lane) : 0u;
  const int e = un.w & 31, n = (un.w >> 5) & 1 ? e : (e + 1) * (e + 2) / 2;
  h.rank = lane < n ? __ldg(R.ranks + un.z + lane) : 0;
  return h;
}

// The pairs of an output tile of degree E whose smaller tile has degree D1: a
// unit's pairs are sorted by it, so a run of one degree is one dispatch.
template <int E, int D1, class Row>
__device__ __forceinline__ void tile_run(const Row& s, uint32_t mine, int m, int& k, uint32_t w,
                                         p2 (&acc)[tri_size(E)]) {
  for (;;) {
    tile_pair<D1, E - D1>(s, (w & 0x1fff) * 2, ((w >> 13) & 0x1fff) * 2, acc);
    if (k + 1 >= m) break;
    w = __shfl_sync(0xffffffffu, mine, k + 1);
    if ((w >> 26) != D1) break;
    ++k;
  }
}

// An output tile of degree E of a warp's 32 items.  Returns its first output.
template <int E, bool TRUNC, class Row>
__device__ __forceinline__ p2 tile_unit(const SquareTable& R, const UnitHead& hd, const Row& s,
                                        const SquareOut& out, p2& rem) {
  const int lane = threadIdx.x & 31;
  const int4 un = hd.un;
  const int diag = (un.w >> 6) & 1, in_n = (un.w >> 8) & 31;
  const int in_off = 2 * ((un.w >> 16) & 0x1fff);
  const int n_off = un.y - diag;             // words of off-diagonal pairs end here
  uint32_t mine = hd.words;
  p2 acc[tri_size(E)];
#pragma unroll
  for (int i = 0; i < tri_size(E); ++i) acc[i] = 0ull;
  for (int k0 = un.x; k0 < n_off; k0 += 32) {
    const uint32_t next = k0 + 32 + lane < un.y ? __ldg(R.words + k0 + 32 + lane) : 0u;
    const int m = min(32, n_off - k0);
    for (int k = 0; k < m; ++k) {
      const uint32_t w = __shfl_sync(0xffffffffu, mine, k);
      const int d1 = w >> 26;
      if (d1 == 0)
        tile_run<E, 0>(s, mine, m, k, w, acc);
      else if (E >= 2 && d1 == 1)
        tile_run<E, (E >= 2 ? 1 : 0)>(s, mine, m, k, w, acc);
      else if (E >= 4 && d1 == 2)
        tile_run<E, (E >= 4 ? 2 : 0)>(s, mine, m, k, w, acc);
    }
    if (k0 + 32 < un.y) mine = next;         // the diagonal's word may be the next chunk's first
  }
  if constexpr (E % 2 == 0)
    if (diag)
      tile_diag<E / 2>(s, 2 * (__shfl_sync(0xffffffffu, mine, (n_off - un.x) & 31) & 0x1fff), acc);
  // in_n: degree + 1 of the input tile of the same prefix (0: none)
  p2 first = 0ull;
#pragma unroll
  for (int r = 0; r <= E; ++r) {
    const int in_row = in_off + pad_row(in_n - 1, r);
#pragma unroll
    for (int c = 0; c <= E - r; c += 2) {
      ulonglong2 lin = make_ulonglong2(0ull, 0ull);
      if (r + c < in_n) lin = s.two(in_row + c);   // a row's padding holds zeros
      const p2 v = put<TRUNC>(out, acc[tri_row(E, r) + c], lin.x,
                              __shfl_sync(0xffffffffu, hd.rank, tri_row(E, r) + c), rem);
      if (r == 0 && c == 0) first = v;
      if (c + 1 <= E - r)
        put<TRUNC>(out, acc[tri_row(E, r) + (c + 1 <= E - r ? c + 1 : c)], lin.y,
                   __shfl_sync(0xffffffffu, hd.rank, tri_row(E, r) + c + 1), rem);
    }
  }
  return first;
}

// One unit (an output tile or row) of a warp's 32 items.  Returns its first
// output (of unit 0: the constant, which the caller finishes).
template <bool TRUNC, class Row>
__device__ __forceinline__ p2 square_unit(const SquareTable& R, const UnitHead& hd, const Row& s,
                                          const SquareOut& out, p2& rem) {
  const int lane = threadIdx.x & 31;
  const int4 un = hd.un;
  const int e = un.w & 31, diag = (un.w >> 6) & 1, in_n = (un.w >> 8) & 31;
  const int in_off = 2 * ((un.w >> 16) & 0x1fff);
  const int n_off = un.y - diag;
  uint32_t mine = hd.words;
  p2 first = 0ull;
  if (!((un.w >> 5) & 1)) {
    switch (e) {
      case 0: return tile_unit<0, TRUNC>(R, hd, s, out, rem);
      case 1: return tile_unit<1, TRUNC>(R, hd, s, out, rem);
      case 2: return tile_unit<2, TRUNC>(R, hd, s, out, rem);
      case 3: return tile_unit<3, TRUNC>(R, hd, s, out, rem);
      case 4: return tile_unit<4, TRUNC>(R, hd, s, out, rem);
      case 5: return tile_unit<5, TRUNC>(R, hd, s, out, rem);
      default: break;
    }
  } else {
    p2 acc[kRowAcc];
#pragma unroll
    for (int i = 0; i < kRowAcc; ++i) acc[i] = 0ull;
    for (int k0 = un.x; k0 < un.y; k0 += 32) {
      const uint32_t next = k0 + 32 + lane < un.y ? __ldg(R.words + k0 + 32 + lane) : 0u;
      const int m = min(32, un.y - k0);
      for (int k = 0; k < m; ++k) {
        const uint32_t w = __shfl_sync(0xffffffffu, mine, k);
        const int o1 = 2 * (w & 0x1fff), o2 = 2 * ((w >> 13) & 0x1fff);
        if (k0 + k < n_off) {
          switch (w >> 26) {
            BERN_ROW_CASES
            default: break;
          }
        } else {
          switch (w >> 26) {
            BERN_RD(1) BERN_RD(2) BERN_RD(3) BERN_RD(4) BERN_RD(5)
            default: break;
          }
        }
      }
      mine = next;
    }
    // e: length of the output row; in_n: of the input row of the same prefix
#pragma unroll
    for (int c = 0; c < 2 * kRowLen - 1; c += 2) {
      if (c >= e) break;
      ulonglong2 lin = make_ulonglong2(0ull, 0ull);
      if (c < in_n) lin = s.two(in_off + c);
      const p2 v = put<TRUNC>(out, acc[c], lin.x, __shfl_sync(0xffffffffu, hd.rank, c), rem);
      if (c == 0) first = v;
      if (c + 1 < e) put<TRUNC>(out, acc[c + 1], lin.y, __shfl_sync(0xffffffffu, hd.rank, c + 1), rem);
    }
  }
  return first;
}

// Units first, first + step, .. of a warp's items.  The tables of the next unit
// are loaded while one is worked on (its header one unit earlier still).
template <bool TRUNC, class Row>
__device__ __forceinline__ void square_units(const SquareTable& R, int first, int step,
                                             const Row& s, const SquareOut& out, p2& rem, p2& c0) {
  if (first >= R.n_units) return;
  UnitHead cur = unit_head(R, __ldg(R.units + first));
  int4 un = __ldg(R.units + min(first + step, R.n_units - 1));
  for (int u = first; u < R.n_units; u += step) {
    const UnitHead nxt = unit_head(R, un);
    un = __ldg(R.units + min(u + 2 * step, R.n_units - 1));
    const p2 v = square_unit<TRUNC>(R, cur, s, out, rem);
    if (u == 0) c0 = v;
    cur = nxt;
  }
}

// The item of a lane: bounds, coefficients and scaling of its group's queue
// entry idx of degree D.
struct SquareItem {
  int64_t item;
  bool valid;
  float Lo, inv, a0, a1, a2;
  int Mpre;
};
__device__ __forceinline__ SquareItem square_item(const ComposeArgs& A, const ComposeScratch& S,
                                                  int D, int idx, int* status) {
  SquareItem it;
  it.valid = idx < S.qcount[D];
  it.item = it.valid ? S.queue[(int64_t)D * S.qcap + idx] : 0;
  it.Lo = it.valid ? A.lo[it.item] : -1.0f;
  it.inv = 1.0f / ((it.valid ? A.hi[it.item] : 1.0f) - it.Lo);
  it.a0 = it.a1 = it.a2 = 0.0f;
  it.Mpre = 0;
  if (it.valid) {
    const float* cf = A.coef + it.item * kCoefStride;
    it.a0 = cf[0];
    it.a1 = cf[1];
    it.a2 = cf[2];
    it.Mpre = A.pre_nterms[it.item];
    if (it.a2 < 0.0f) atomicOr(status, kStatusUnsupported);   // excluded by convexity
  }
  return it;
}
__device__ __forceinline__ SquareOut square_out(const Tables& T, const ComposeArgs& A,
                                                const SquareItem& it, int D) {
  const int64_t to = A.base(it.item, A.post_ld);
  return SquareOut{A.post_up + to, A.post_lo + to, A.h, pack2(-it.a1, it.a1),
                   pack2(it.a2, it.a2), T.mcount[min(2 * D, A.cap)], it.valid};
}

// s = (pre - lo*[K=0]) / (hi - lo) in round-to-nearest of one bound (P), ranks
// in groups of eight: groups first, first + step, ..; the pair at position p of
// the lane starts at dst[4 (p / 2) stride + 2 (p % 2)].  The padding gets
// zeros.  Returns sum|s| of them (rounded up).
__device__ __forceinline__ float load_s(const ComposeArgs& A, const SquareTable& R,
                                        const SquareItem& it, const float* P, int first, int step,
                                        float* dst, int stride) {
  const int h = A.h;
  P += A.base(it.item, A.pre_ld);
  float l1 = 0.0f;
  for (int r0 = 8 * first; r0 < R.m_pad; r0 += 8 * step) {
    float v[8];
    int pos[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int r = r0 + i;                  // from m_in on: padding positions
      v[i] = r < it.Mpre ? __ldg(P + (int64_t)r * h) : 0.0f;
      pos[i] = r < R.m_pad ? __ldg(R.pos + r) : -1;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (pos[i] < 0) continue;
      float x = v[i];
      if (r0 + i == 0) x = __fsub_rn(x, it.Lo);
      x = __fmul_rn(x, it.inv);
      dst[4 * (int64_t)(pos[i] >> 1) * stride + 2 * (pos[i] & 1)] = x;
      l1 = __fadd_ru(l1, fabsf(x));
    }
  }
  return l1;
}

// Constant term: a0 + (its value without a0) + Lip*eta + remainder.
__device__ __forceinline__ void put_constant(const ComposeArgs& A, const SquareItem& it,
                                             const SquareOut& o, p2 c0, p2 l1, p2 rem,
                                             int* status) {
  float l1l, l1u, rl, ru, cl, cu;
  unpack2(l1, l1l, l1u);
  unpack2(rem, rl, ru);
  unpack2(c0, cl, cu);
  const float eu = __fmul_ru(5.0f * kU, l1u), el = __fmul_ru(5.0f * kU, l1l);
  const float lu = __fmaf_ru(2.0f * it.a2, __fadd_ru(1.0f, eu), fabsf(it.a1));
  const float ll = __fmaf_ru(2.0f * it.a2, __fadd_ru(1.0f, el), fabsf(it.a1));
  const float vu = __fadd_ru(__fadd_ru(__fadd_ru(cu, it.a0), __fmul_ru(lu, eu)), ru);
  float vl = __fsub_rd(__fadd_rd(-cl, it.a0), __fmul_ru(ll, el));
  vl = __fadd_rd(__fsub_rd(vl, A.eps[it.item]), -rl);
  o.QU[0] = vu;
  o.QL[0] = vl;
  if (!isfinite(vu) || !isfinite(vl)) atomicOr(status, kStatusNonFinite);
}

// The degree and 32-item group of task `task` among the queues dlo..dhi, or
// D = -1 past the last.
__device__ __forceinline__ int find_group(const ComposeScratch& S, int dlo, int dhi, int& group) {
  for (int d = dlo; d <= dhi; ++d) {
    const int nc = (S.qcount[d] + 31) >> 5;
    if (group < nc) return d;
    group -= nc;
  }
  return -1;
}

// Inputs in shared memory, WPG warps to a group: they share the loads and then the
// units in turn.  A block per group for long inputs or few groups, fewer warps for
// short inputs of many groups (down to one, without barriers).
constexpr int kSquareWarps = 8;
constexpr int kSquareBlocks = 2;
constexpr int kLoadParts = 4;                // partial sums of |s| (as the fused layer's)

template <int WPG>
__device__ __forceinline__ void group_sync(int group) {
  if constexpr (WPG == kSquareWarps)
    __syncthreads();
  else if constexpr (WPG > 1)
    asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "n"(32 * WPG) : "memory");
  else
    __syncwarp();
}

template <int WPG>
__global__ void __launch_bounds__(32 * kSquareWarps, kSquareBlocks)
k_square(Tables T, ComposeArgs A, ComposeScratch S, int dlo, int dhi, int sstride, int* status) {
  static_assert(2 * kLoadParts % WPG == 0, "the loads of both bounds over the warps of a group");
  constexpr int GPB = kSquareWarps / WPG;    // groups of a block
  extern __shared__ __align__(16) p2 smem2[];
  __shared__ float s_l1[WPG > 1 ? GPB : 1][2][kLoadParts][32];
  __shared__ p2 s_rem[kSquareWarps][32], s_c0[GPB][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, w = warp % WPG, g = warp / WPG;
  p2* mine = smem2 + (size_t)(32 * g + lane) * sstride;
  for (int task = blockIdx.x * GPB + g;; task += gridDim.x * GPB) {
    int group = task;
    const int D = find_group(S, dlo, dhi, group);
    if (D < 0) break;
    const SquareTable R = T.sqt[D];
    const SquareItem it = square_item(A, S, D, group * 32 + lane, status);
    p2 l1 = 0ull;
    if constexpr (WPG > 1) {
#pragma unroll
      for (int i = 0; i < 2 * kLoadParts / WPG; ++i) {
        const int k = w + i * WPG, up = k / kLoadParts, part = k - up * kLoadParts;
        s_l1[g][up][part][lane] = load_s(A, R, it, up ? A.pre_up : A.pre_lo, part, kLoadParts,
                                         reinterpret_cast<float*>(mine) + up, 1);
      }
    } else {
#pragma unroll
      for (int part = 0; part < kLoadParts; ++part) {
        const float u = load_s(A, R, it, A.pre_up, part, kLoadParts,
                               reinterpret_cast<float*>(mine) + 1, 1);
        const float l = load_s(A, R, it, A.pre_lo, part, kLoadParts,
                               reinterpret_cast<float*>(mine), 1);
        l1 = part == 0 ? pack2(l, u) : add2_ru(l1, pack2(l, u));
      }
    }
    group_sync<WPG>(g);
    const SquareOut out = square_out(T, A, it, D);
    p2 rem = 0ull, c0 = 0ull;
    if (2 * D <= A.cap)
      square_units<false>(R, w, WPG, SmemRow{mine}, out, rem, c0);
    else
      square_units<true>(R, w, WPG, SmemRow{mine}, out, rem, c0);
    if constexpr (WPG > 1) {
      s_rem[warp][lane] = rem;
      if (w == 0) s_c0[g][lane] = c0;        // unit 0 holds the constant
      group_sync<WPG>(g);
      if (w == 0) {
        l1 = pack2(s_l1[g][0][0][lane], s_l1[g][1][0][lane]);
#pragma unroll
        for (int i = 1; i < kLoadParts; ++i)
          l1 = add2_ru(l1, pack2(s_l1[g][0][i][lane], s_l1[g][1][i][lane]));
#pragma unroll
        for (int i = 1; i < WPG; ++i) rem = add2_ru(rem, s_rem[warp + i][lane]);
        if (it.valid) put_constant(A, it, out, s_c0[g][lane], l1, rem, status);
      }
    } else {
      if (it.valid) put_constant(A, it, out, c0, l1, rem, status);
    }
    group_sync<WPG>(g);                      // the next task reuses the shared inputs
  }
}

// Inputs beyond shared memory, three kernels over the groups
// [first, first + groups) of the queues dlo..dhi: s to the scratch (a block per
// group), the units of a group in kSquareChunks interleaved parts over blocks, and
// the constant terms from the parts' remainders in order.
//   scratch of a group: padded pairs x 32 lanes of s, then per warp of the parts a
//   remainder (32 pairs), the constant and sum|s| (32 pairs each).
// The units kernel waits for its loads of s (14 resident warps, a third of them from
// the L1): one block of 16 warps on neighbouring units per multiprocessor instead
// of two of 8 shares more of the L1, and 16 tasks per group of its size end closer
// together (100 groups, n = 6, D = 8: 7.1 ms, 6.9 with 8 tasks, 6.4 with 16 and
// 6.3 with 32, whose remainders cost that again).
constexpr int kSquareWarpTerms = 32;         // padded terms of a warp per group
constexpr int kSquarePairTerms = 50;         // of two warps per group
constexpr int kSquareFewTerms = 12;
constexpr int kSquareChunks = 16;
constexpr int kUnitWarps = 16;                // one block per multiprocessor
constexpr int kSquareParts = kSquareChunks * kUnitWarps;

__global__ void __launch_bounds__(256)
k_square_scale(Tables T, ComposeArgs A, ComposeScratch S, int dlo, int dhi, int first, int groups,
               int64_t gstride, int* status) {
  __shared__ float s_l1[2][4][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int g = blockIdx.x; g < groups; g += gridDim.x) {
    int group = first + g;
    const int D = find_group(S, dlo, dhi, group);
    if (D < 0) break;
    const SquareTable R = T.sqt[D];
    const SquareItem it = square_item(A, S, D, group * 32 + lane, status);
    p2* base = reinterpret_cast<p2*>(S.tws) + (int64_t)g * gstride;
    const int up = warp >> 2, part = warp & 3;
    s_l1[up][part][lane] = load_s(A, R, it, up ? A.pre_up : A.pre_lo, part, 4,
                                  reinterpret_cast<float*>(base + 2 * lane) + up, 32);
    __syncthreads();
    if (warp == 0) {
      p2 l1 = pack2(s_l1[0][0][lane], s_l1[1][0][lane]);
#pragma unroll
      for (int w = 1; w < 4; ++w) l1 = add2_ru(l1, pack2(s_l1[0][w][lane], s_l1[1][w][lane]));
      base[gstride - 32 + lane] = l1;
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(32 * kUnitWarps, 1)
k_square_units(Tables T, ComposeArgs A, ComposeScratch S, int dlo, int dhi, int first, int groups,
               int64_t gstride, int* status) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int task = blockIdx.x; task < groups * kSquareChunks; task += gridDim.x) {
    const int g = task / kSquareChunks, part = (task - g * kSquareChunks) * kUnitWarps + warp;
    int group = first + g;
    const int D = find_group(S, dlo, dhi, group);
    if (D < 0) break;
    const SquareTable R = T.sqt[D];
    const SquareItem it = square_item(A, S, D, group * 32 + lane, status);
    p2* base = reinterpret_cast<p2*>(S.tws) + (int64_t)g * gstride;
    const SquareOut out = square_out(T, A, it, D);
    p2 rem = 0ull, c0 = 0ull;
    const ScratchRow s{base + 2 * lane};
    if (2 * D <= A.cap)
      square_units<false>(R, part, kSquareParts, s, out, rem, c0);
    else
      square_units<true>(R, part, kSquareParts, s, out, rem, c0);
    p2* tail = base + gstride - (kSquareParts + 2) * 32;
    tail[part * 32 + lane] = rem;
    if (part == 0) tail[kSquareParts * 32 + lane] = c0;   // unit 0 holds the constant
  }
}

__global__ void __launch_bounds__(32)
k_square_constant(Tables T, ComposeArgs A, ComposeScratch S, int dlo, int dhi, int first,
                  int groups, int64_t gstride, int* status) {
  const int lane = threadIdx.x;
  for (int g = blockIdx.x; g < groups; g += gridDim.x) {
    int group = first + g;
    const int D = find_group(S, dlo, dhi, group);
    if (D < 0) break;
    const SquareItem it = square_item(A, S, D, group * 32 + lane, status);
    const p2* tail = reinterpret_cast<const p2*>(S.tws) + (int64_t)(g + 1) * gstride -
                     (kSquareParts + 2) * 32;
    p2 rem = 0ull;
    for (int part = 0; part < kSquareParts; ++part) rem = add2_ru(rem, tail[part * 32 + lane]);
    if (it.valid)
      put_constant(A, it, square_out(T, A, it, D), tail[kSquareParts * 32 + lane],
                   tail[(kSquareParts + 1) * 32 + lane], rem, status);
  }
}

// pairs of a group's scratch slice for inputs of m padded terms
int64_t group_pairs(int64_t m) { return 32 * (m + kSquareParts + 2); }

}  // namespace

int square_smem_degree(int n) {
  int D = kMaxRowDegree;
  while (D > 0 && num_monomials(n, D) > kSquareSmemTerms) --D;
  return D;
}
int square_max_degree(int n) {
  int D = kMaxRowDegree;
  while (D > 0 && num_monomials(n, D) > kSquareMaxTerms) --D;
  return D;
}

size_t square_group_bytes(int n, int Dmax) {
  const int D = std::min(Dmax, square_max_degree(n));
  if (D <= square_smem_degree(n)) return 0;
  return (size_t)group_pairs(square_padded_terms(n, D)) * sizeof(p2);
}
size_t square_scratch_bytes(int n, int Dmax, int64_t n_items, int64_t limit) {
  const int64_t per = (int64_t)square_group_bytes(n, Dmax);
  if (per == 0) return 0;
  // a group may be short, one per degree
  const int64_t groups = (n_items + 31) / 32 + kMaxRowDegree;
  return (size_t)(per * std::min<int64_t>(groups, limit / per));
}

cudaError_t launch_compose_square(const Launch& L, const Tables& T, const ComposeScratch& S,
                                  const ComposeArgs& A, int64_t n_items, int Dmax) {
  const int dsm = std::min(std::min(Dmax, T.sqt_dmax), square_smem_degree(T.n));
  const int dmx = std::min(std::min(Dmax, T.sqt_dmax), square_max_degree(T.n));
  // A warp per group where every input of the layer is short and there is a group
  // for every resident warp: order 2 on degree 2 in three variables, 327,680
  // items, 41 us with a block per group, 26 us.
  const int pad = square_padded_terms(T.n, dsm);
  const int64_t resident = (int64_t)32 * kSquareWarps * kSquareBlocks * device_sms(L);
  const bool one = pad <= kSquareWarpTerms && n_items >= resident;
  // Two warps for inputs about as long (degrees 7 and 8 in two variables, 4 in three),
  // whose 13 to 17 units eight warps share badly: degree 8 in two variables, 327,680
  // items of which 1/5, 1/2 and all are squared in place, 8 / 4 / 2 / 1 warps a group
  // (us): 151 / 146 / 149 / 168, 220 / 193 / 184 / 199, 347 / 278 / 237 / 238.  From
  // seven eighths of the resident warps on (70,400 items, all: 83 / - / 64; 44,800,
  // 1/3: 33 / 30 / 40), inputs of a few units already from half of them on (degree 2 in
  // two variables, 44,800 items, all: 27 / - / 17 / 15 us; 19,200, 2/5: 14.5 / - / 14.7),
  // and where the cap keeps all outputs: the sum over the others has a part per warp.
  const bool two = !one && pad <= kSquarePairTerms && 2 * dsm <= A.cap &&
                   n_items >= (pad <= kSquareFewTerms ? resident / 2 : resident / 8 * 7);
  auto launch = [&](auto kern, int wpg, int dlo, int dhi) -> cudaError_t {
    // the per-lane stride is an odd number of 16-byte units, so that lanes
    // reading the same position hit distinct banks
    const int sstride = square_padded_terms(T.n, dhi) | 2, gpb = kSquareWarps / wpg;
    const size_t smem = (size_t)32 * gpb * sstride * sizeof(p2);
    if (smem > 40 * 1024) {
      const cudaError_t e =
          cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
    }
    const int64_t tasks = (n_items / 32 + (dhi - dlo) + 1 + gpb - 1) / gpb;
    kern<<<(unsigned)std::min<int64_t>(tasks, device_sms(L) * kSquareBlocks), 32 * kSquareWarps,
           smem, L.stream>>>(T, A, S, dlo, dhi, sstride, L.status);
    ++*L.launches;
    return cudaGetLastError();
  };
  const cudaError_t e = one   ? launch(k_square<1>, 1, 0, dsm)
                        : two ? launch(k_square<2>, 2, 0, dsm)
                              : launch(k_square<kSquareWarps>, kSquareWarps, 0, dsm);
  if (e != cudaSuccess) return e;
  if (dmx > dsm && S.tws) {
    const int64_t gstride = group_pairs(square_padded_terms(T.n, dmx));
    const int64_t fit = S.tws_bytes / (gstride * (int64_t)sizeof(p2));
    if (fit < 1) return cudaErrorInvalidValue;
    const int64_t all = n_items / 32 + (dmx - dsm) + 1;
    for (int64_t first = 0; first < all; first += fit) {
      const int groups = (int)std::min<int64_t>(fit, all - first);
      k_square_scale<<<(unsigned)std::min<int64_t>(groups, device_sms(L) * 8), 256, 0, L.stream>>>(
          T, A, S, dsm + 1, dmx, (int)first, groups, gstride, L.status);
      k_square_units<<<(unsigned)std::min<int64_t>((int64_t)groups * kSquareChunks,
                                                   device_sms(L) * 8),
                       32 * kUnitWarps, 0, L.stream>>>(T, A, S, dsm + 1, dmx, (int)first,
                                                         groups, gstride, L.status);
      k_square_constant<<<(unsigned)std::min<int64_t>(groups, device_sms(L) * 16), 32, 0,
                          L.stream>>>(T, A, S, dsm + 1, dmx, (int)first, groups, gstride,
                                      L.status);
      *L.launches += 3;
    }
  }
  return cudaGetLastError();
}

}  // namespace bern
