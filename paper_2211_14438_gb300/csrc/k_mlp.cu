// The learned component's kernels: degree features, BF16 MLP inference,
// the cross-entropy gradient (deterministic two-pass reduction) and Adam.
//
// Forward, per sample (one thread), weights staged in shared memory:
//   xb = bf16(x);  for each hidden unit j:  z1_j = b1_j + sum_f W1_jf xb_f,
//   a_j = bf16(max(z1_j, 0)),  z_c += W2_cj a_j  (fp32 accumulation).
// Backward:  p = softmax(z),  dz_c = w (p_c - [c = y]),
//   dW2_cj = sum_s dz_c a_j,  db2_c = sum_s dz_c,
//   dz1_j = [z1_j > 0] sum_c W2_cj dz_c,  dW1_jf = sum_s dz1_j xb_f,  db1_j = sum_s dz1_j,
// all divided by n.  A block keeps the sums of its tiles of samples in registers
// (per-sample terms live in shared memory only); a second kernel adds the blocks'
// sums in block order, so the result does not depend on scheduling.
#include <math.h>

#include <algorithm>

#include "device_util.cuh"
#include "enclose_impl.cuh"
#include "mlp.cuh"

namespace bern {

namespace {

constexpr int kH = kMlpHidden;

struct SmemMlp {
  float W1[kH * kMlpMaxF];     // [j][f], zero-padded to kMlpMaxF
  float b1[kH];
  float W2[kMlpMaxC * kH];     // [c][j]
  float b2[kMlpMaxC];
};

__device__ void stage_mlp(const MlpView& M, SmemMlp& S) {
  for (int i = threadIdx.x; i < kH * kMlpMaxF; i += blockDim.x) {
    const int j = i / kMlpMaxF, f = i % kMlpMaxF;
    S.W1[i] = f < M.F ? __bfloat162float(M.W1[j * M.F + f]) : 0.0f;
  }
  for (int i = threadIdx.x; i < kH; i += blockDim.x) S.b1[i] = M.b1[i];
  for (int i = threadIdx.x; i < kMlpMaxC * kH; i += blockDim.x)
    S.W2[i] = i < M.C * kH ? __bfloat162float(M.W2[i]) : 0.0f;
  for (int i = threadIdx.x; i < kMlpMaxC; i += blockDim.x) S.b2[i] = i < M.C ? M.b2[i] : 0.0f;
  __syncthreads();
}

__device__ __forceinline__ float bf16_round(float v) {
  return __bfloat162float(__float2bfloat16_rn(v));
}

__device__ __forceinline__ float hidden_pre(const SmemMlp& S, int j, const float (&xb)[kMlpMaxF]) {
  float acc = S.b1[j];
#pragma unroll
  for (int f = 0; f < kMlpMaxF; ++f) acc = fmaf(S.W1[j * kMlpMaxF + f], xb[f], acc);
  return acc;
}

// Logits of one sample.
__device__ void mlp_logits(const SmemMlp& S, const float (&xb)[kMlpMaxF], float (&z)[kMlpMaxC]) {
#pragma unroll
  for (int c = 0; c < kMlpMaxC; ++c) z[c] = S.b2[c];
  for (int j = 0; j < kH; ++j) {
    const float a = bf16_round(fmaxf(hidden_pre(S, j, xb), 0.0f));
#pragma unroll
    for (int c = 0; c < kMlpMaxC; ++c) z[c] = fmaf(S.W2[c * kH + j], a, z[c]);
  }
}

__device__ void load_features(const float* x, int F, int64_t s, float (&xb)[kMlpMaxF]) {
#pragma unroll
  for (int f = 0; f < kMlpMaxF; ++f) xb[f] = f < F ? bf16_round(x[s * F + f]) : 0.0f;
}

__global__ void __launch_bounds__(128)
k_degree_features(int64_t n, const float* __restrict__ lo, const float* __restrict__ hi,
                  const int32_t* __restrict__ nterms, int layer, float* __restrict__ x) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    float f[kDegFeatures];
    degree_feature_vec(lo[i], hi[i], nterms ? nterms[i] : 1, layer, f);
#pragma unroll
    for (int k = 0; k < kDegFeatures; ++k) x[i * kDegFeatures + k] = f[k];
  }
}

// The proposals of a box by a warp, two neurons per lane at a time.  Weights in
// shared memory at the proposals' own sizes (8 features, 4 classes), four values
// per load, each load for both neurons; the products and their order are those
// of mlp_logits, whose padding only adds zeros.
//
// Bound: FMA issue and the shared loads that feed it (half each).  A block of 128
// threads per box at the padded sizes took 39 us for 5120 boxes of 64 neurons,
// this 25 us.
static_assert(kDegFeatures <= 8 && kDegClasses <= 4, "proposal weights are two and one float4");

__global__ void __launch_bounds__(128)
k_learned_degrees(MlpView M, int64_t n_boxes, int h, int layer, const float* __restrict__ lo,
                  const float* __restrict__ hi, const int32_t* __restrict__ pre_nterms,
                  float min_conf, int fallback_d, int max_d, int cap,
                  const int32_t* __restrict__ order_in,
                  int32_t* __restrict__ order_out, uint8_t* __restrict__ degrees,
                  int8_t* __restrict__ kind, float* __restrict__ coef, float* __restrict__ eps,
                  int* status) {
  __shared__ float4 s_w1[kH][2], s_w2[kH];
  __shared__ float s_b1[kH], s_b2[4];
  for (int i = threadIdx.x; i < kH * 8; i += blockDim.x) {
    const int j = i >> 3, f = i & 7;
    reinterpret_cast<float*>(s_w1)[i] =
        f < kDegFeatures ? __bfloat162float(M.W1[j * kDegFeatures + f]) : 0.0f;
  }
  for (int i = threadIdx.x; i < kH * 4; i += blockDim.x) {
    const int j = i >> 2, c = i & 3;
    reinterpret_cast<float*>(s_w2)[i] = c < kDegClasses ? __bfloat162float(M.W2[c * kH + j]) : 0.0f;
  }
  for (int i = threadIdx.x; i < kH; i += blockDim.x) s_b1[i] = M.b1[i];
  if (threadIdx.x < 4) s_b2[threadIdx.x] = threadIdx.x < kDegClasses ? M.b2[threadIdx.x] : 0.0f;
  __syncthreads();
  const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  for (int64_t b = (int64_t)blockIdx.x * warps + (threadIdx.x >> 5); b < n_boxes;
       b += (int64_t)gridDim.x * warps) {
    int dmax = 1;
    for (int m = lane; m < h; m += 64) {
      float l[2], u[2], xb[2][8], z[2][4];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int64_t it = b * h + min(m + 32 * q, h - 1);
        l[q] = lo[it];
        u[q] = hi[it];
        float f[kDegFeatures];
        degree_feature_vec(l[q], u[q], pre_nterms[it], layer, f);
#pragma unroll
        for (int k = 0; k < 8; ++k) xb[q][k] = k < kDegFeatures ? bf16_round(f[k]) : 0.0f;
#pragma unroll
        for (int c = 0; c < 4; ++c) z[q][c] = s_b2[c];
      }
#pragma unroll 4
      for (int j = 0; j < kH; ++j) {
        const float4 wa = s_w1[j][0], wb = s_w1[j][1], v = s_w2[j];
        const float w[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
        const float v4[4] = {v.x, v.y, v.z, v.w};
        const float b1 = s_b1[j];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          float acc = b1;
#pragma unroll
          for (int k = 0; k < 8; ++k) acc = fmaf(w[k], xb[q][k], acc);
          const float a = bf16_round(fmaxf(acc, 0.0f));
#pragma unroll
          for (int c = 0; c < 4; ++c) z[q][c] = fmaf(v4[c], a, z[q][c]);
        }
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        if (m + 32 * q >= h) continue;
        const int64_t it = b * h + m + 32 * q;
        int best = 0;
        float zb = z[q][0];
#pragma unroll
        for (int c = 1; c < kDegClasses; ++c)
          if (z[q][c] > zb) {   // first maximum wins ties
            zb = z[q][c];
            best = c;
          }
        float sum = 0.0f;
#pragma unroll
        for (int c = 0; c < kDegClasses; ++c) sum += expf(z[q][c] - zb);
        const float conf = 1.0f / sum;   // the largest softmax probability
        const int d = min(conf >= min_conf ? best + 1 : fallback_d, max_d);
        degrees[it] = (uint8_t)d;
        kind[it] = (int8_t)relu_item(l[q], u[q], d, coef + it * kCoefStride, eps + it, status);
        dmax = max(dmax, d);
      }
    }
    __syncwarp();
    dmax = warp_imax(dmax);
    if (lane == 0) order_out[b] = min(cap, order_in[b] * dmax);
  }
}

__global__ void k_fill_i32(int32_t* p, int64_t n, int32_t v) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    p[i] = v;
}

__global__ void __launch_bounds__(128)
k_mlp_forward(MlpView M, int64_t n, const float* __restrict__ x, float* __restrict__ logits) {
  __shared__ SmemMlp S;
  stage_mlp(M, S);
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n;
       s += (int64_t)gridDim.x * blockDim.x) {
    float xb[kMlpMaxF], z[kMlpMaxC];
    load_features(x, M.F, s, xb);
    mlp_logits(S, xb, z);
#pragma unroll
    for (int c = 0; c < kMlpMaxC; ++c)
      if (c < M.C) logits[s * M.C + c] = z[c];
  }
}

// Backward: a block takes tiles of kTile samples in turn.  First four lanes share
// a sample (lane part p has the hidden units 4 i + p) and leave the tile's
// activations, hidden and logit gradients in shared memory, one row per unit;
// then thread (j, p) adds the tile to its parameters: W1[j][f] of a quarter of
// the features, W2[c][j] of c = p, p + 4, and the biases.
//
// Bound: instruction issue (about 120 warp instructions per sample).  Through
// memory (a [n][64] gradient and activation array written by strided stores and
// read back by a thread per parameter, serially over 1024 samples) 204,800
// samples took 174 + 336 + 27 us; now 72 + 7 us.
constexpr int kTile = 64;
constexpr int kTileStride = kTile + 8;   // rows on 16 bytes; four rows on distinct banks
constexpr int kBackThreads = 4 * kTile;
constexpr int kBackBlocks = 512;         // most blocks (partial sums)
static_assert(kBackThreads == 4 * kH, "a thread per (unit, part)");

constexpr int kBackPerSM = 3;            // resident blocks (85 registers, 44-51 KB)
template <int FP, int CP>
__global__ void __launch_bounds__(kBackThreads, kBackPerSM)
k_mlp_back(MlpView M, int64_t n, const float* __restrict__ x, const int32_t* __restrict__ labels,
           const float* __restrict__ w, float* __restrict__ partial, int64_t P, int* status) {
  __shared__ float sW1[kH][FP], sb1[kH], sW2[CP][kH], sb2[CP];
  __shared__ __align__(16) float sX[FP][kTileStride], sD1[kH][kTileStride], sA[kH][kTileStride],
      sD2[CP][kTileStride];
  __shared__ float sLoss[kTile];
  const int tid = threadIdx.x, part = tid & 3, F = M.F, C = M.C;
  for (int i = tid; i < kH * FP; i += kBackThreads) {
    const int j = i / FP, f = i - j * FP;
    sW1[j][f] = f < F ? __bfloat162float(M.W1[j * F + f]) : 0.0f;
  }
  for (int i = tid; i < kH; i += kBackThreads) sb1[i] = M.b1[i];
  for (int i = tid; i < CP * kH; i += kBackThreads)
    sW2[i / kH][i % kH] = i < C * kH ? __bfloat162float(M.W2[i]) : 0.0f;
  if (tid < CP) sb2[tid] = tid < C ? M.b2[tid] : 0.0f;
  for (int i = tid; i < FP * kTileStride; i += kBackThreads) (&sX[0][0])[i] = 0.0f;
  float gW1[FP / 4], gW2[CP / 4], gb1 = 0.0f, gb2[CP / 4], gl = 0.0f;
#pragma unroll
  for (int i = 0; i < FP / 4; ++i) gW1[i] = 0.0f;
#pragma unroll
  for (int i = 0; i < CP / 4; ++i) gW2[i] = gb2[i] = 0.0f;
  const int64_t tiles = (n + kTile - 1) / kTile;
  for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const int64_t s0 = t * kTile;
    const int have = (int)min((int64_t)kTile, n - s0);
    __syncthreads();                       // the previous tile is added
    for (int i = tid; i < kTile * F; i += kBackThreads) {
      const int s = i / F, f = i - s * F;
      sX[f][s] = s < have ? bf16_round(x[s0 * F + i]) : 0.0f;
    }
    __syncthreads();
    {
      const int s = tid >> 2;
      const bool live = s < have;
      float xb[FP], z[CP];
      unsigned on = 0;                     // the units with a positive input
#pragma unroll
      for (int f = 0; f < FP; ++f) xb[f] = sX[f][s];
#pragma unroll
      for (int c = 0; c < CP; ++c) z[c] = 0.0f;
#pragma unroll 4
      for (int i = 0; i < kH / 4; ++i) {
        const int j = 4 * i + part;
        float pre = sb1[j];
#pragma unroll
        for (int f = 0; f < FP; ++f) pre = fmaf(sW1[j][f], xb[f], pre);
        const float a = bf16_round(fmaxf(pre, 0.0f));
        sA[j][s] = a;
        on |= (pre > 0.0f ? 1u : 0u) << i;
#pragma unroll
        for (int c = 0; c < CP; ++c) z[c] = fmaf(sW2[c][j], a, z[c]);
      }
      float mx = -INFINITY;
#pragma unroll
      for (int c = 0; c < CP; ++c) {
        z[c] += __shfl_xor_sync(0xffffffffu, z[c], 1);
        z[c] += __shfl_xor_sync(0xffffffffu, z[c], 2);
        z[c] += sb2[c];
        if (c < C) mx = fmaxf(mx, z[c]);
      }
      float e[CP], sum = 0.0f;
#pragma unroll
      for (int c = 0; c < CP; ++c) {
        e[c] = c < C ? expf(z[c] - mx) : 0.0f;
        sum += e[c];
      }
      int y = live ? labels[s0 + s] : 0;
      float ws = live ? (w ? w[s0 + s] : 1.0f) : 0.0f;
      if (y < 0 || y >= C) {
        if (part == 0) atomicOr(status, kStatusInvalid);
        y = 0;
        ws = 0.0f;
      }
      float zy = 0.0f;
#pragma unroll
      for (int c = 0; c < CP; ++c)
        if (c == y) zy = z[c];
      const float inv = 1.0f / sum;
#pragma unroll
      for (int c = 0; c < CP; ++c) {
        e[c] = c < C && live ? ws * (e[c] * inv - (c == y ? 1.0f : 0.0f)) : 0.0f;   // dz_c
        if ((c & 3) == part) sD2[c][s] = e[c];
      }
      if (part == 0) sLoss[s] = live ? ws * (logf(sum) - (zy - mx)) : 0.0f;
#pragma unroll 4
      for (int i = 0; i < kH / 4; ++i) {
        const int j = 4 * i + part;
        float dh = 0.0f;
#pragma unroll
        for (int c = 0; c < CP; ++c) dh = fmaf(sW2[c][j], e[c], dh);
        sD1[j][s] = (on >> i) & 1 ? dh : 0.0f;
      }
    }
    __syncthreads();
    const int j = tid >> 2;
#pragma unroll 2
    for (int s = 0; s < kTile; s += 4) {
      const float4 d = *reinterpret_cast<const float4*>(&sD1[j][s]);
      const float4 av = *reinterpret_cast<const float4*>(&sA[j][s]);
#pragma unroll
      for (int i = 0; i < FP / 4; ++i) {
        const float4 v = *reinterpret_cast<const float4*>(&sX[part * (FP / 4) + i][s]);
        gW1[i] = fmaf(d.x, v.x, gW1[i]);
        gW1[i] = fmaf(d.y, v.y, gW1[i]);
        gW1[i] = fmaf(d.z, v.z, gW1[i]);
        gW1[i] = fmaf(d.w, v.w, gW1[i]);
      }
#pragma unroll
      for (int i = 0; i < CP / 4; ++i) {
        const float4 g = *reinterpret_cast<const float4*>(&sD2[part + 4 * i][s]);
        gW2[i] = fmaf(g.x, av.x, gW2[i]);
        gW2[i] = fmaf(g.y, av.y, gW2[i]);
        gW2[i] = fmaf(g.z, av.z, gW2[i]);
        gW2[i] = fmaf(g.w, av.w, gW2[i]);
        gb2[i] += g.x + g.y + (g.z + g.w);
      }
      gb1 += d.x + d.y + (d.z + d.w);
      if (tid == 0) gl += sLoss[s] + sLoss[s + 1] + (sLoss[s + 2] + sLoss[s + 3]);
    }
  }
  // this block's sums (parameter order: W1, b1, W2, b2, then the loss)
  float* out = partial + (int64_t)blockIdx.x * (P + 1);
  const int j = tid >> 2;
  const int64_t ob1 = (int64_t)kH * F, oW2 = ob1 + kH, ob2 = oW2 + (int64_t)C * kH;
#pragma unroll
  for (int i = 0; i < FP / 4; ++i) {
    const int f = part * (FP / 4) + i;
    if (f < F) out[j * F + f] = gW1[i];
  }
  if (part == 0) out[ob1 + j] = gb1;
#pragma unroll
  for (int i = 0; i < CP / 4; ++i) {
    const int c = part + 4 * i;
    if (c < C) {
      out[oW2 + c * kH + j] = gW2[i];
      if (j == 0) out[ob2 + c] = gb2[i];
    }
  }
  if (tid == 0) out[P] = gl;
}

// The blocks' sums of 32 parameters: eight slices of blocks, each in order,
// added in order.
__global__ void __launch_bounds__(256)
k_mlp_back_final(int64_t n, int64_t P, int blocks, const float* __restrict__ partial,
                 float* __restrict__ grad, float* __restrict__ loss) {
  __shared__ float s_sum[8][32];
  const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
  const int64_t p = (int64_t)blockIdx.x * 32 + lane;
  const int per = (blocks + 7) / 8, c0 = slice * per, c1 = min(blocks, c0 + per);
  float acc = 0.0f;
  if (p <= P) {
#pragma unroll 8
    for (int c = c0; c < c1; ++c) acc += partial[(int64_t)c * (P + 1) + p];
  }
  s_sum[slice][lane] = acc;
  __syncthreads();
  if (slice == 0 && p <= P) {
#pragma unroll
    for (int k = 1; k < 8; ++k) acc += s_sum[k][lane];
    const float v = acc / (float)n;
    if (p < P)
      grad[p] = v;
    else
      loss[0] = v;
  }
}

__global__ void __launch_bounds__(256)
k_mlp_adam(int F, int C, int64_t P, float* __restrict__ param, float* __restrict__ m,
           float* __restrict__ v, const float* __restrict__ grad, float lr, float beta1,
           float beta2, float eps, float c1, float c2, __nv_bfloat16* __restrict__ W1b,
           __nv_bfloat16* __restrict__ W2b) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= P) return;
  const float g = grad[p];
  const float mm = beta1 * m[p] + (1.0f - beta1) * g;
  const float vv = beta2 * v[p] + (1.0f - beta2) * g * g;
  m[p] = mm;
  v[p] = vv;
  const float th = param[p] - lr * (mm / c1) / (sqrtf(vv / c2) + eps);
  param[p] = th;
  const int64_t oW1 = (int64_t)kH * F, ob1 = oW1 + kH, oW2 = ob1 + (int64_t)C * kH;
  if (p < oW1) W1b[p] = __float2bfloat16_rn(th);
  else if (p >= ob1 && p < oW2) W2b[p - ob1] = __float2bfloat16_rn(th);
}

}  // namespace

size_t mlp_backward_scratch(int64_t n, int F, int C) {
  const int64_t blocks = std::min<int64_t>(kBackBlocks, (n + kTile - 1) / kTile);
  return sizeof(float) * (size_t)std::max<int64_t>(1, blocks) * (size_t)(mlp_num_params(F, C) + 1);
}

static unsigned grid_for(int64_t n, int threads, int cap) {
  int64_t g = (n + threads - 1) / threads;
  if (g < 1) g = 1;
  return (unsigned)(g < cap ? g : cap);
}

cudaError_t launch_degree_features(const Launch& L, int64_t n_items, const float* lo,
                                   const float* hi, const int32_t* nterms, int layer, float* x) {
  if (n_items == 0) return cudaSuccess;
  k_degree_features<<<grid_for(n_items, 128, device_sms(L) * 32), 128, 0, L.stream>>>(n_items, lo, hi,
                                                                           nterms, layer, x);
  ++*L.launches;
  return cudaGetLastError();
}

cudaError_t launch_learned_degrees(const Launch& L, const MlpView& M, int64_t n_boxes, int h,
                                   int layer, const float* lo, const float* hi,
                                   const int32_t* pre_nterms, float min_conf, int fallback_d,
                                   int max_d, int cap, const int32_t* order_in,
                                   int32_t* order_out, uint8_t* degrees, int8_t* kind,
                                   float* coef, float* eps) {
  if (n_boxes == 0) return cudaSuccess;
  if (M.F != kDegFeatures || M.C != kDegClasses) return cudaErrorInvalidValue;
  k_learned_degrees<<<grid_for(n_boxes, 4, device_sms(L) * 16), 128, 0, L.stream>>>(
      M, n_boxes, h, layer, lo, hi, pre_nterms, min_conf, fallback_d, max_d, cap, order_in,
      order_out,
      degrees, kind, coef, eps, L.status);
  ++*L.launches;
  return cudaGetLastError();
}

cudaError_t launch_fill_i32(const Launch& L, int32_t* p, int64_t n, int32_t v) {
  if (n == 0) return cudaSuccess;
  k_fill_i32<<<grid_for(n, 256, device_sms(L) * 8), 256, 0, L.stream>>>(p, n, v);
  ++*L.launches;
  return cudaGetLastError();
}

cudaError_t launch_mlp_forward(const Launch& L, const MlpView& M, int64_t n, const float* x,
                               float* logits) {
  if (n == 0) return cudaSuccess;
  k_mlp_forward<<<grid_for(n, 128, device_sms(L) * 16), 128, 0, L.stream>>>(M, n, x, logits);
  ++*L.launches;
  return cudaGetLastError();
}

cudaError_t launch_mlp_backward(const Launch& L, const MlpView& M, int64_t n, const float* x,
                                const int32_t* labels, const float* w, void* scratch,
                                float* grad, float* loss) {
  if (n <= 0) return cudaErrorInvalidValue;
  const int64_t P = mlp_num_params(M.F, M.C);
  float* partial = (float*)scratch;
  const int blocks = (int)std::min<int64_t>(std::min<int64_t>(kBackBlocks, kBackPerSM * device_sms(L)),
                                            (n + kTile - 1) / kTile);
  auto kern = M.F <= 8 ? (M.C <= 4 ? k_mlp_back<8, 4> : k_mlp_back<8, 8>)
                       : (M.C <= 4 ? k_mlp_back<16, 4> : k_mlp_back<16, 8>);
  kern<<<blocks, kBackThreads, 0, L.stream>>>(M, n, x, labels, w, partial, P, L.status);
  k_mlp_back_final<<<(unsigned)((P + 1 + 31) / 32), 256, 0, L.stream>>>(n, P, blocks, partial,
                                                                        grad, loss);
  *L.launches += 2;
  return cudaGetLastError();
}

cudaError_t launch_mlp_adam(const Launch& L, int F, int C, float* param, float* m, float* v,
                            const float* grad, float lr, float beta1, float beta2, float eps,
                            float c1, float c2, __nv_bfloat16* W1b, __nv_bfloat16* W2b) {
  const int64_t P = mlp_num_params(F, C);
  k_mlp_adam<<<(unsigned)((P + 255) / 256), 256, 0, L.stream>>>(F, C, P, param, m, v, grad, lr,
                                                                 beta1, beta2, eps, c1, c2, W1b,
                                                                 W2b);
  ++*L.launches;
  return cudaGetLastError();
}

}  // namespace bern
