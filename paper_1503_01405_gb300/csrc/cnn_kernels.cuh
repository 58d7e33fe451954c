// Kernels of the single-pulse candidate classifier (see cnn.cu for the network).
//
// Layout: activations [B][C][T] (C = 32 DM-trial channels), BF16 in memory
// between layers, FP32 in registers and shared memory; every sum accumulates
// in FP32.  Weight gradients are formed per sample and reduced over the batch
// in sample order, so a training step is deterministic.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace pond {
namespace cnn {

constexpr int C = 32;          // channels
constexpr int K = 7;           // kernel width
constexpr int PAD = 3;
constexpr int T0 = 256;        // samples per patch
constexpr int NCLS = 4;
constexpr int CONV = C * C * K;                       // 7168 weights per conv layer
constexpr int LAYER = CONV + C;                       // weights + biases
constexpr int FC_OFF = 3 * LAYER;                     // 21,600
constexpr int NPARAM = FC_OFF + NCLS * C + NCLS;      // 21,732
constexpr int THREADS = 256;

__device__ __forceinline__ float bf(const __nv_bfloat16 v) { return __bfloat162float(v); }

// The conv kernels of a layer of T samples give a thread four rows (output
// channels, or input channels in the backward pass) of eight consecutive samples: per input row
// it reads a window of 16 samples and 28 weights (11 16-byte shared-memory loads) for 224
// multiply-adds.  A CTA of 128 threads holds half of the rows (blockIdx.y) of SPB =
// 256 / T samples, so a batch of 256 is 3.4 CTAs per SM at T = 256.  With a thread per
// row and 32 samples, read one by one from rows that met in the same banks, the passes kept the
// shared-memory pipe 51-70 % busy at 17-24 % issue.  Batch 256: forward 166 -> 60 us,
// backward data 60 -> 37 us, weight gradients 69 -> 62 us (and the weights staged
// from a copy in the kernels' own order: the whole step 233 -> 200 us).
constexpr int CT = 128;                               // threads
constexpr int HALF = C / 2;                           // rows per CTA
template <int T> __host__ __device__ constexpr int spb() { return 256 / T; }
template <int T> __host__ __device__ constexpr int xpitch() { return T + 12; }   // 3 zeros, T samples, zeros; 4 mod 32
template <int T> constexpr int conv_smem_bytes() {
  return (spb<T>() * C * xpitch<T>() + C * K * HALF) * (int)sizeof(float);
}

// Rows of SPB samples as FP32 with PAD zeros ahead (sample t of row r at r pitch + t +
// PAD): load(b, r, t) gives four consecutive samples.
template <int T, class Load>
__device__ __forceinline__ void stage_rows(float* xs, int b0, int B, Load load) {
  constexpr int P = xpitch<T>(), Q = T / 4;
  for (int i = threadIdx.x; i < spb<T>() * C * 8; i += CT) {   // the 8 samples of each row outside 0 .. T-1
    const int r = i >> 3, e = i & 7;
    xs[r * P + (e < PAD ? e : T + e)] = 0.f;
  }
#pragma unroll 8
  for (int i = threadIdx.x; i < spb<T>() * C * Q; i += CT) {
    const int r = i / Q, t = 4 * (i % Q), b = b0 + r / C;
    const float4 v = b < B ? load(b, r % C, t) : make_float4(0.f, 0.f, 0.f, 0.f);
    float* d = xs + r * P + t + PAD;
    d[0] = v.x;
    d[1] = v.y;
    d[2] = v.z;
    d[3] = v.w;
  }
}

// Four consecutive BF16 values (8-byte aligned unless ANY).
template <bool ANY>
__device__ __forceinline__ float4 load_bf4(const __nv_bfloat16* p) {
  if constexpr (ANY) {
    return make_float4(bf(p[0]), bf(p[1]), bf(p[2]), bf(p[3]));
  } else {
    const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16),
                       __uint_as_float(u.y & 0xffff0000u));
  }
}

// The FP32 copies of the conv weights the kernels above read, made after every parameter
// update: layer l, forward [half of co][ci][k][HALF co], then backward [half of ci][co][k][HALF ci].
constexpr int WHALF = C * K * HALF, WCONV = 2 * WHALF;      // floats per half, per direction of a layer
constexpr int WF_FLOATS = 3 * 2 * WCONV;
__global__ void k_conv_weights(const __nv_bfloat16* __restrict__ wbf, float* __restrict__ wf) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 3 * CONV) return;
  const int l = i / CONV, r = i % CONV, co = r / (C * K), ci = (r / K) % C, k = r % K;
  const float v = bf(wbf[l * LAYER + r]);
  float* o = wf + l * 2 * WCONV;
  o[(co / HALF) * WHALF + (ci * K + k) * HALF + co % HALF] = v;
  o[WCONV + (ci / HALF) * WHALF + (co * K + k) * HALF + ci % HALF] = v;
}

__device__ __forceinline__ void stage_weights(float* ws, const float* __restrict__ wf) {
  static_assert(WHALF % (4 * CT) == 0, "whole rounds");
#pragma unroll
  for (int u = 0; u < WHALF / (4 * CT); ++u) {
    const int i = threadIdx.x + u * CT;
    reinterpret_cast<float4*>(ws)[i] = __ldg(reinterpret_cast<const float4*>(wf) + i);
  }
}

// acc[r][i] += sum over the C input rows and the K taps, in that order, of weight (row r,
// input row, tap) times the window's sample i + tap (the taps in reverse for REV).
// ws: [input row][tap][HALF] floats.
template <int T, bool REV>
__device__ __forceinline__ void conv_tile(const float* xs, const float* ws, int rg, int t0, float (&acc)[4][8]) {
  constexpr int P = xpitch<T>();
#pragma unroll 1
  for (int ci = 0; ci < C; ++ci) {
    float x[16];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 v = *reinterpret_cast<const float4*>(xs + ci * P + t0 + 4 * q);
      x[4 * q] = v.x;
      x[4 * q + 1] = v.y;
      x[4 * q + 2] = v.z;
      x[4 * q + 3] = v.w;
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const float4 w = *reinterpret_cast<const float4*>(ws + (ci * K + k) * HALF + 4 * rg);
      const float wr[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[r][i] = fmaf(wr[r], x[i + (REV ? 2 * PAD - k : k)], acc[r][i]);
    }
  }
}

// Forward conv: z = b + w * x (zero padded), a = relu(z).
// MODE 0: 2:1 max-pool of a -> out (BF16) and the argmax of each pair; MODE 1:
// global average of a over time -> gap (FP32).  z is kept for the backward pass.
// ANYX: x need not be 8-byte aligned.
template <int T, int MODE, bool ANYX>
__global__ void __launch_bounds__(CT) k_conv_fwd(const __nv_bfloat16* __restrict__ x,
                                                 const float* __restrict__ wf, const float* __restrict__ bias,
                                                 int B, float* __restrict__ z, __nv_bfloat16* __restrict__ out,
                                                 uint8_t* __restrict__ arg, float* __restrict__ gap) {
  extern __shared__ float4 sm4[];
  float* xs = reinterpret_cast<float*>(sm4);
  float* ws = xs + spb<T>() * C * xpitch<T>();
  const int b0 = blockIdx.x * spb<T>(), co0 = blockIdx.y * HALF;
  stage_rows<T>(xs, b0, B, [&](int b, int r, int t) { return load_bf4<ANYX>(x + ((size_t)b * C + r) * T + t); });
  stage_weights(ws, wf + blockIdx.y * WHALF);
  __syncthreads();
  constexpr int TG = T / 8;                          // time groups: 4 TG threads per sample
  const int tid = threadIdx.x, s = tid / (4 * TG), rg = (tid / TG) & 3, tg = tid % TG, b = b0 + s;
  float acc[4][8];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[r][i] = bias[co0 + 4 * rg + r];
  conv_tile<T, false>(xs + s * C * xpitch<T>(), ws, rg, 8 * tg, acc);
  if (b < B) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const size_t row = (size_t)b * C + co0 + 4 * rg + r;
      float4* zb = reinterpret_cast<float4*>(z + row * T + 8 * tg);
      zb[0] = make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
      zb[1] = make_float4(acc[r][4], acc[r][5], acc[r][6], acc[r][7]);
      if constexpr (MODE == 0) {
        __nv_bfloat162 h[2];
        uchar4 a;
        float m[4];
        unsigned char q[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float a0 = fmaxf(acc[r][2 * i], 0.f), a1 = fmaxf(acc[r][2 * i + 1], 0.f);
          m[i] = a1 > a0 ? a1 : a0;
          q[i] = a1 > a0 ? 1 : 0;
        }
        h[0] = __floats2bfloat162_rn(m[0], m[1]);
        h[1] = __floats2bfloat162_rn(m[2], m[3]);
        a = make_uchar4(q[0], q[1], q[2], q[3]);
        const size_t o = row * (T / 2) + 4 * tg;
        *reinterpret_cast<uint2*>(out + o) =
            make_uint2(*reinterpret_cast<const uint32_t*>(&h[0]), *reinterpret_cast<const uint32_t*>(&h[1]));
        *reinterpret_cast<uchar4*>(arg + o) = a;
      }
    }
  }
  if constexpr (MODE == 1) {
    // sums of eight samples, then the time groups in order
    __syncthreads();                                 // the staged rows are read
    float* part = xs;                                // [sample][row][TG]
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      float t = 0.f;
#pragma unroll
      for (int i = 0; i < 8; ++i) t += fmaxf(acc[r][i], 0.f);
      part[(s * HALF + 4 * rg + r) * TG + tg] = t;
    }
    __syncthreads();
    for (int i = tid; i < spb<T>() * HALF; i += CT) {
      float g = 0.f;
#pragma unroll
      for (int q = 0; q < TG; ++q) g += part[i * TG + q];
      if (b0 + i / HALF < B) gap[(size_t)(b0 + i / HALF) * C + co0 + i % HALF] = g / (float)T;
    }
  }
}

// Head of one sample per warp: logits = fc_w g + fc_b, softmax, per-sample
// cross-entropy, d loss / d logits (scaled by 1/B for the batch mean), dg, and
// the fc gradient partials of this sample.  Lane j < NCLS forms logit j, its sum over the
// channels in order; lane c owns channel c of the rest.
__global__ void __launch_bounds__(128) k_head(const float* __restrict__ gap, const __nv_bfloat16* __restrict__ fcw,
                                              const float* __restrict__ fcb, const int32_t* __restrict__ labels, int B,
                                              float* __restrict__ prob, float* __restrict__ loss,
                                              float* __restrict__ dg, float* __restrict__ part) {
  static_assert(C == 32, "a lane per channel");
  const int b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (b >= B) return;
  const float g = gap[(size_t)b * C + lane];
  float wc[NCLS], lg[NCLS];
#pragma unroll
  for (int j = 0; j < NCLS; ++j) {
    wc[j] = bf(fcw[j * C + lane]);
    lg[j] = fcb[j];
  }
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const float gc = __shfl_sync(0xffffffffu, g, c);
#pragma unroll
    for (int j = 0; j < NCLS; ++j) lg[j] = fmaf(__shfl_sync(0xffffffffu, wc[j], c), gc, lg[j]);
  }
  float mx = -INFINITY, den = 0.f;
#pragma unroll
  for (int j = 0; j < NCLS; ++j) mx = fmaxf(mx, lg[j]);
#pragma unroll
  for (int j = 0; j < NCLS; ++j) {
    lg[j] = expf(lg[j] - mx);
    den += lg[j];
  }
#pragma unroll
  for (int j = 0; j < NCLS; ++j) lg[j] /= den;
#pragma unroll
  for (int j = 0; j < NCLS; ++j)
    if (lane == j) prob[(size_t)b * NCLS + j] = lg[j];
  if (!labels) return;
  const int y = labels[b];
  float ly = lg[0], dl[NCLS];
#pragma unroll
  for (int j = 0; j < NCLS; ++j) {
    if (j == y) ly = lg[j];
    dl[j] = (lg[j] - (j == y ? 1.f : 0.f)) / (float)B;
  }
  if (lane == 0) loss[b] = -logf(fmaxf(ly, 1e-30f));
  float* pb = part + (size_t)b * NPARAM + FC_OFF;
  float s = 0.f;
#pragma unroll
  for (int j = 0; j < NCLS; ++j) {
    pb[j * C + lane] = dl[j] * g;
    s = fmaf(dl[j], wc[j], s);
    if (lane == j) pb[NCLS * C + j] = dl[j];
  }
  dg[(size_t)b * C + lane] = s;
}

// Four consecutive values of a layer's dz: stored, or (AVG, the last layer) the
// backward of the global average, (z > 0) dg / T.
template <int T, bool AVG>
__device__ __forceinline__ float4 load_dz(const float* __restrict__ dz, const float* __restrict__ dg, size_t row, int t) {
  const float4 v = __ldg(reinterpret_cast<const float4*>(dz + row * T + t));
  if constexpr (!AVG) return v;
  const float d = dg[row] / (float)T;
  return make_float4(v.x > 0.f ? d : 0.f, v.y > 0.f ? d : 0.f, v.z > 0.f ? d : 0.f, v.w > 0.f ? d : 0.f);
}

// Backward data pass of a conv layer of length T:
// dh[ci][t] = sum_{co,k} w[co][ci][k] dz[co][t + PAD - k], then the previous
// layer's max-pool and ReLU are undone: dz_prev[ci][2t + arg] = dh (z_prev > 0).
// AVG: dz holds the layer's z and dg its global average's gradient.
template <int T, bool AVG>
__global__ void __launch_bounds__(CT) k_conv_bwd_data(const float* __restrict__ dz, const float* __restrict__ dg,
                                                      const float* __restrict__ wf,
                                                      const uint8_t* __restrict__ arg_prev,
                                                      const float* __restrict__ z_prev, int B,
                                                      float* __restrict__ dz_prev) {
  extern __shared__ float4 sm4[];
  float* ds = reinterpret_cast<float*>(sm4);
  float* ws = ds + spb<T>() * C * xpitch<T>();
  const int b0 = blockIdx.x * spb<T>(), ci0 = blockIdx.y * HALF;
  stage_rows<T>(ds, b0, B, [&](int b, int r, int t) { return load_dz<T, AVG>(dz, dg, (size_t)b * C + r, t); });
  stage_weights(ws, wf + blockIdx.y * WHALF);
  __syncthreads();
  constexpr int TG = T / 8;
  const int tid = threadIdx.x, s = tid / (4 * TG), rg = (tid / TG) & 3, tg = tid % TG, b = b0 + s;
  float acc[4][8];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[r][i] = 0.f;
  conv_tile<T, true>(ds + s * C * xpitch<T>(), ws, rg, 8 * tg, acc);
  if (b >= B) return;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const size_t row = (size_t)b * C + ci0 + 4 * rg + r, t = 8 * tg;
    const uint2 a2 = __ldg(reinterpret_cast<const uint2*>(arg_prev + row * T + t));
    const float4* zp = reinterpret_cast<const float4*>(z_prev + row * (2 * T) + 2 * t);
    float4* dp = reinterpret_cast<float4*>(dz_prev + row * (2 * T) + 2 * t);
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
      const unsigned aw = i < 4 ? a2.x : a2.y;
      const bool a0 = (aw >> (8 * (i & 3))) & 1u, a1 = (aw >> (8 * (i & 3) + 8)) & 1u;
      const float4 zv = __ldg(zp + i / 2);
      dp[i / 2] = make_float4(!a0 && zv.x > 0.f ? acc[r][i] : 0.f, a0 && zv.y > 0.f ? acc[r][i] : 0.f,
                              !a1 && zv.z > 0.f ? acc[r][i + 1] : 0.f, a1 && zv.w > 0.f ? acc[r][i + 1] : 0.f);
    }
  }
}

// Per-sample weight and bias gradients of a conv layer of length T:
// dW[co][ci][k] = sum_t dz[co][t] x[ci][t + k - PAD], db[co] = sum_t dz[co][t],
// written to this sample's row of the partials at offset `off`.  A thread holds 4 x 4 channel
// pairs and all taps (112 sums) over a quarter of the samples; the quarters are added in
// order through shared memory.
constexpr int WT = 256;
template <int T> __host__ __device__ constexpr int wpitch() { return T + 4; }      // dz rows
template <int T> constexpr int wgt_smem_bytes() {
  constexpr int a = C * (wpitch<T>() + xpitch<T>()) * (int)sizeof(float), b = 3 * 64 * 113 * (int)sizeof(float);
  return a > b ? a : b;
}
template <int T, bool ANYX, bool AVG>
__global__ void __launch_bounds__(WT) k_conv_bwd_weight(const float* __restrict__ dz, const float* __restrict__ dg,
                                                        const __nv_bfloat16* __restrict__ x, float* __restrict__ part,
                                                        int off) {
  extern __shared__ float4 sm4[];
  constexpr int DP = wpitch<T>(), P = xpitch<T>(), Q = T / 4;
  float* ds = reinterpret_cast<float*>(sm4);          // [C][DP]
  float* xs = ds + C * DP;                            // [C][P]: sample t at t + PAD
  const int b = blockIdx.x, tid = threadIdx.x;
  for (int i = tid; i < C * 8; i += WT) xs[(i >> 3) * P + ((i & 7) < PAD ? (i & 7) : T + (i & 7))] = 0.f;
  for (int i = tid; i < C * Q; i += WT) {
    const int r = i / Q, t = 4 * (i % Q);
    const size_t row = (size_t)b * C + r;
    *reinterpret_cast<float4*>(ds + r * DP + t) = load_dz<T, AVG>(dz, dg, row, t);
    const float4 v = load_bf4<ANYX>(x + row * T + t);
    float* d = xs + r * P + t + PAD;
    d[0] = v.x;
    d[1] = v.y;
    d[2] = v.z;
    d[3] = v.w;
  }
  __syncthreads();
  const int quarter = tid >> 6, cog = (tid >> 3) & 7, cig = tid & 7;   // channels cog + 8 r, cig + 8 s
  float acc[4][4][K];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int k = 0; k < K; ++k) acc[r][s][k] = 0.f;
  float bias[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
  for (int t = quarter * (T / 4); t < (quarter + 1) * (T / 4); t += 4) {
    float d[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float4 v = *reinterpret_cast<const float4*>(ds + (cog + 8 * r) * DP + t);
      d[r][0] = v.x;
      d[r][1] = v.y;
      d[r][2] = v.z;
      d[r][3] = v.w;
#pragma unroll
      for (int i = 0; i < 4; ++i) bias[r] += d[r][i];
    }
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      float xw[12];                                   // samples t - PAD .. t + 8
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const float4 v = *reinterpret_cast<const float4*>(xs + (cig + 8 * s) * P + t + 4 * q);
        xw[4 * q] = v.x;
        xw[4 * q + 1] = v.y;
        xw[4 * q + 2] = v.z;
        xw[4 * q + 3] = v.w;
      }
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int k = 0; k < K; ++k) acc[r][s][k] = fmaf(d[r][i], xw[i + k], acc[r][s][k]);
    }
  }
  __syncthreads();                                    // the rows are read
  float* red = ds;                                    // [quarter - 1][64][113]
  if (quarter) {
    float* o = red + ((quarter - 1) * 64 + (tid & 63)) * 113;
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int k = 0; k < K; ++k) o[(r * 4 + s) * K + k] = acc[r][s][k];
  }
  __syncthreads();
  float* pb = part + (size_t)b * NPARAM + off;
  if (!quarter) {
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const float* o = red + (q * 64 + tid) * 113;
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
          for (int k = 0; k < K; ++k) acc[r][s][k] += o[(r * 4 + s) * K + k];
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int k = 0; k < K; ++k) pb[((cog + 8 * r) * C + cig + 8 * s) * K + k] = acc[r][s][k];
  }
  __syncthreads();                                    // the quarters are added
  if (cig == 0)
#pragma unroll
    for (int r = 0; r < 4; ++r) red[quarter * C + cog + 8 * r] = bias[r];
  __syncthreads();
  if (tid < C) pb[CONV + tid] = (red[tid] + red[C + tid]) + (red[2 * C + tid] + red[3 * C + tid]);
}

// grad[p] = sum over samples b of part[b][p]: four consecutive quarters of the batch, each in
// order, added in order; the last CTA takes the mean loss (every 256th loss per
// thread, then a fixed tree).
constexpr int RT = 256, RP = RT / 4, REDUCE_BLOCKS = (NPARAM + RP - 1) / RP;
__global__ void __launch_bounds__(RT) k_reduce(const float* __restrict__ part, const float* __restrict__ loss, int B,
                                               float* __restrict__ grad, float* __restrict__ lmean) {
  __shared__ float red[RT];
  const int tid = threadIdx.x;
  if (blockIdx.x == REDUCE_BLOCKS) {
    float s = 0.f;
    for (int b = tid; b < B; b += RT) s += loss[b];
    red[tid] = s;
    for (int h = RT / 2; h > 0; h >>= 1) {
      __syncthreads();
      if (tid < h) red[tid] += red[tid + h];
    }
    if (tid == 0) *lmean = red[0] / (float)B;
    return;
  }
  const int q = tid / RP, p = blockIdx.x * RP + tid % RP, per = (B + 3) / 4;
  float s = 0.f;
  if (p < NPARAM)
#pragma unroll 16
    for (int b = q * per; b < min(B, (q + 1) * per); ++b) s += __ldg(part + (size_t)b * NPARAM + p);
  red[tid] = s;
  __syncthreads();
  if (q == 0 && p < NPARAM) grad[p] = ((red[tid] + red[tid + RP]) + red[tid + 2 * RP]) + red[tid + 3 * RP];
}

// Adam (Kingma & Ba 2015) on the FP32 master weights; refreshes the BF16 copy.
__global__ void k_adam(float* __restrict__ theta, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ grad, __nv_bfloat16* __restrict__ wbf, float lr, float c1,
                       float c2, float beta1, float beta2, float eps) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= NPARAM) return;
  const float g = grad[p];
  const float mm = beta1 * m[p] + (1.f - beta1) * g;
  const float vv = beta2 * v[p] + (1.f - beta2) * g * g;
  m[p] = mm;
  v[p] = vv;
  const float th = theta[p] - lr * (mm / c1) / (sqrtf(vv / c2) + eps);
  theta[p] = th;
  wbf[p] = __float2bfloat16(th);
}

// Patch p: trials d0..d0+C-1, samples t0..t0+T0-1 of a series block
// [ndm][stride] (samples outside [0, n) repeat the nearest edge sample), less
// its mean and over its standard deviation (1 when that is zero), as BF16.
__global__ void __launch_bounds__(THREADS) k_patches(const float* __restrict__ series, int ndm, long long n,
                                                     long long stride, const int32_t* __restrict__ corner,
                                                     __nv_bfloat16* __restrict__ out) {
  __shared__ float red[THREADS];
  __shared__ float stat[2];
  const int p = blockIdx.x;
  const int d0 = corner[2 * p];
  const long long t0 = corner[2 * p + 1];
  constexpr int NV = C * T0 / THREADS;
  float v[NV];
  float s = 0.f;
#pragma unroll
  for (int u = 0; u < NV; ++u) {
    const int i = threadIdx.x + u * THREADS;
    const int d = min(max(d0 + i / T0, 0), ndm - 1);
    const long long t = min(max(t0 + i % T0, 0ll), n - 1);
    v[u] = series[(size_t)d * stride + t];
    s += v[u];
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int h = THREADS / 2; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) stat[0] = red[0] / (float)(C * T0);
  __syncthreads();
  const float mean = stat[0];
  s = 0.f;
#pragma unroll
  for (int u = 0; u < NV; ++u) s += (v[u] - mean) * (v[u] - mean);
  __syncthreads();
  red[threadIdx.x] = s;
  __syncthreads();
  for (int h = THREADS / 2; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const float sd = sqrtf(red[0] / (float)(C * T0));
    stat[1] = sd > 0.f ? sd : 1.f;
  }
  __syncthreads();
  const float inv = 1.f / stat[1];
#pragma unroll
  for (int u = 0; u < NV; ++u)
    out[(size_t)p * C * T0 + threadIdx.x + u * THREADS] = __float2bfloat16((v[u] - mean) * inv);
}

}  // namespace cnn
}  // namespace pond
